// Incidence construction: r-clique -> s-clique incidence as CSR (Def. 1).
//
// The paper discovers the s-cliques of an r-clique through the
// neighbourhoods of its vertices (Section 4.1, "Time complexity": all
// (s-r)-tuples of a neighbourhood), and recomputes them on every pass.  Here
// they are found once, by sorted-list intersection, and stored:
//   (1,2)  the CSR itself is the incidence (q = 1), under ids ordered by
//          degree class for graphs of 65,536 vertices or more;
//   (2,3)  triangle {u,v,w} -> one pair per edge: the CSR slots of its other
//          two edges at the edge's endpoints (found once each, by degree
//          orientation), each row then ordered by the third vertex;
//   (3,4)  triangle (u,v,w): the z in the triangle lists of its three edges
//          -> the slots of {u,v,z}, {u,w,z}, {v,w,z} in those lists.
// Every step is a count pass, an exclusive scan and a fill pass over the same
// enumeration; the (2,3) fill of larger graphs takes the count's triangles as
// records.  Intersections: (2,3), 32 oriented edges per warp, the elements of
// their shorter out-lists walked as one sequence and binary-searched in the
// longer ones; (3,4), a list pair or triple per warp, the longer lists passing
// through shared memory in blocks (nd_list_cursor) or, where much longer,
// binary-searched.
#include "nd_internal.cuh"

#include <vector>

namespace {

constexpr int kThreads = 256;
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t* __restrict__ a, int64_t lo,
                                                   int64_t hi, int32_t x) {
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (__ldg(a + mid) < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ unsigned lanemask_lt() {
    return (1u << (threadIdx.x & 31)) - 1u;
}

__device__ __forceinline__ int64_t warp_id_global() {
    return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}

__device__ __forceinline__ int64_t warp_count_global() {
    return ((int64_t)gridDim.x * blockDim.x) >> 5;
}

// ---- 32 rows per warp ------------------------------------------------------
// Most rows of these graphs hold fewer entries than a warp has lanes.  The
// kernels below therefore give a warp up to 32 consecutive rows: lane l loads what
// leads to row l, and the entries of all are then walked as one sequence,
// 32 at a time (row_pool).  Rows of more than kPoolRow entries go to
// a second walk, one at a time and spread over all warps: consecutive rows are
// of like length (degree classes, the edges of one hub), and 32 long ones would
// keep one warp busy long after the others.  (A warp per row spent a chain of loads
// on every row, empty ones included: 30 of the 97 ms of a batch of 256 small
// graphs went to such kernels.)
constexpr int kPoolRow = 128;
// Rows per warp: 32 where that still gives every resident warp some, fewer
// otherwise (a 2,800-vertex graph validated in 37 instead of 18 us with 32).
int rows_per_warp(const nd_incidence* h, int64_t rows) {
    const int64_t r = rows / ((h->sm_count > 0 ? h->sm_count : 152) * 64);
    return (int)(r < 1 ? 1 : (r > 32 ? 32 : r));
}
int pool_blocks(int64_t rows, int per, int cap) { return nd_blocks_for((rows + per - 1) / per * 32, kThreads, cap); }

// the rows of [0, n) for which pick(row) holds, spread over the warps: f(row)
template <typename P, typename F>
__device__ __forceinline__ void spread_rows(int64_t n, P&& pick, F&& f) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = warp_count_global();
    for (int64_t first = warp_id_global(); first < n; first += 32 * warps) {
        const int64_t mine = first + lane * warps;
        for (unsigned todo = __ballot_sync(kFull, mine < n && pick(mine)); todo; todo &= todo - 1)
            f(first + (__ffs(todo) - 1) * warps);
    }
}

struct row_pool {
    struct place {
        int row, at;    // the entry's row, and the entries before it
        unsigned same;  // the lanes with entries of that row
    };
    // the warp's words: entries before each row, then of each row that is not
    // empty, in order, the same * 32 + its index (a row has fewer than 2^22)
    uint32_t* pre;
    int total;
    int start;   // the first entry of this lane's row, -1 if it is empty
    int before;  // rows, not empty, that begin before the next block
    static constexpr int kWords = 64;
    // len: entries of this lane's row
    __device__ __forceinline__ row_pool(uint32_t* words, int len) : pre(words), before(0) {
        const int lane = threadIdx.x & 31;
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        const unsigned filled = __ballot_sync(kFull, len > 0);
        __syncwarp();
        pre[lane] = (uint32_t)(incl - len);
        if (len > 0) pre[32 + __popc(filled & lanemask_lt())] = (uint32_t)(incl - len) << 5 | lane;
        start = len > 0 ? incl - len : -1;
        total = __shfl_sync(kFull, incl, 31);
        __syncwarp();
    }
    // where this lane's entry of the block of 32 from e0 lies; blocks are asked
    // for in order, and lanes past the last entry get the last row.  One bit per
    // row that begins in the block, so one shared load finds the row, where a
    // search of the prefix sums takes five in a row (triangle count of the R-MAT
    // k-truss of 1,048,576 vertices: 13.3 against 12.5 ms).
    __device__ __forceinline__ place block(int e0) {
        const int lane = threadIdx.x & 31;
        const unsigned d = (unsigned)(start - e0);
        const unsigned begins = __reduce_or_sync(kFull, d < 32u ? 1u << d : 0u);
        const unsigned upto = 0xffffffffu >> (31 - lane), starts = begins | 1u;
        const uint32_t q = pre[31 + before + __popc(begins & upto)];
        before += __popc(begins);
        const unsigned later = starts & ~upto;
        const unsigned from_first = 0xffffffffu << (31 - __clz(starts & upto));
        return {(int)(q & 31u), (int)(q >> 5), later ? from_first & ((1u << (__ffs(later) - 1)) - 1u) : from_first};
    }
    // the entries of row r
    __device__ __forceinline__ int length(int r) const { return (r < 31 ? (int)pre[r + 1] : total) - (int)pre[r]; }
};

// ---- validation and degree split ------------------------------------------
// A row must lie inside [0, nnz], be strictly increasing and hold ids in
// [0, n) other than its own, and every entry v of row u needs u in row v.
// Writes nlow[u] = #neighbours < u and upcnt[u] = #neighbours > u.  Reads
// only inside the bounds it has checked, so a malformed graph cannot fault.
//
// Symmetry: vertices are ordered by the key (row length, id).  An entry
// (u, v) whose row u has the larger key searches the shorter row v for u;
// the others are not searched.  The reverse of a searching entry is a
// non-searching one, and distinct entries have distinct reverses, so if
// every searching entry finds its reverse and the searching entries are
// exactly half of nnz (counted in *searched, checked by the host), the two
// halves are in one-to-one correspondence: the graph is symmetric.  A hub
// row is thus never binary-searched, whatever the order of the caller's ids.
// BY_LENGTH = false: the key is the id alone, so the entries above the
// diagonal search (the same argument holds).  That is for graphs whose ids
// the build itself assigned by degree class, high degree first, where the
// entry above the diagonal already points at the shorter row (or one of its
// class) and nothing needs gathering to decide it.
// With mirror (builds with r >= 2), it also records for both entries of
// every pair the position of the other: the reverse entry, found by the same
// search.

// FP (k-core builds, which need no reverse entries): symmetry by
// fingerprint instead of searches.  Every entry (u, v) adds +f(u, v), if
// u < v, or -f(v, u) to two 64-bit sums, each with its own mixing function f
// (the splitmix64 finalizer, after Steele, Lea and Flood, and the finalizer of
// its result).  A symmetric graph sums to zero exactly.  Otherwise the sums
// are those of +-f over the entries without a reverse, and both are zero only
// by a coincidence of two 64-bit hashes.  It streams col once and gathers
// nothing; the hashing bounds it, so an entry takes two finalizers (f(u, v) -
// f(v, u) with unrelated inputs took six).
__device__ __forceinline__ unsigned long long fp_mix(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ void fp_add(unsigned long long (&fp)[2], int64_t u, int32_t v) {
    const bool up = u < v;
    const unsigned long long lo = up ? (unsigned long long)u : (unsigned long long)v;
    const unsigned long long hi = up ? (unsigned long long)v : (unsigned long long)u;
    const unsigned long long a = fp_mix(((lo << 32) | hi) ^ 0x9e3779b97f4a7c15ull);
    const unsigned long long b = fp_mix(a + 0x632be59bd9b4e019ull);
    fp[0] += up ? a : 0ull - a;
    fp[1] += up ? b : 0ull - b;
}

// the checks of entries [pb, pe) of row u (which spans [b, e)), one entry
// per lane: the count of entries below the diagonal, of searching entries,
// and whether any check failed (FP: fp collects this lane's fingerprint
// terms, summed over the warp by the caller)
template <bool BY_LENGTH, bool FP>
__device__ __forceinline__ bool validate_entry(int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                               const int32_t* __restrict__ col, int64_t u, int64_t b, int64_t e,
                                               int64_t p, uint32_t* __restrict__ mirror, bool& low, int& found,
                                               unsigned long long (&fp)[2]) {
    const int32_t v = col[p];
    if (v < 0 || v >= n || v == u) return false;
    low = v < u;
    const bool ok = p <= b || col[p - 1] < v;
    if constexpr (FP) {
        fp_add(fp, u, v);
        return ok;
    }
    if (!BY_LENGTH && v < u) return ok;
    const int64_t vb = rp[v], ve = rp[v + 1];
    // a row longer than n - 1 cannot be simple (and would not fit the 32-bit search)
    if (vb < 0 || ve < vb || ve > nnz || ve - vb >= n) return false;
    if (BY_LENGTH && (e - b < ve - vb || (e - b == ve - vb && u < v))) return ok;
    const int64_t pos = vb + nd_lower_bound_n(col + vb, (int)(ve - vb), (int32_t)u);
    if (pos >= ve || col[pos] != (int32_t)u) return false;
    ++found;
    if (mirror) {
        mirror[p] = (uint32_t)pos;
        mirror[pos] = (uint32_t)p;
    }
    return ok;
}

template <bool BY_LENGTH, bool FP = false>
__device__ __forceinline__ void validate_entries(int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                                 const int32_t* __restrict__ col, int64_t u, int64_t b, int64_t e,
                                                 int64_t pb, int64_t pe, uint32_t* __restrict__ mirror, int& low,
                                                 int& found, bool& rowbad, unsigned long long (&fp)[2]) {
    const int lane = threadIdx.x & 31;
    for (int64_t p = pb + lane; p < pe; p += 32) {
        bool below = false;
        if (!validate_entry<BY_LENGTH, FP>(n, nnz, rp, col, u, b, e, p, mirror, below, found, fp)) rowbad = true;
        low += below;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        low += __shfl_xor_sync(kFull, low, o);
        found += __shfl_xor_sync(kFull, found, o);
    }
    rowbad = __any_sync(kFull, rowbad);
}

// Rows longer than kLongRow entries are not walked by one warp (a hub row of
// a million entries would take a single warp tens of thousands of dependent
// steps): the per-vertex kernels skip them, and a second launch spreads
// their kLongSeg-entry segments over the whole grid.
constexpr int64_t kLongRow = 4096;
constexpr int64_t kLongSeg = 1024;

__device__ __forceinline__ bool is_long_row(int64_t b, int64_t e) { return e - b > kLongRow; }

// the rows (with valid bounds) longer than kLongRow, and their lengths.  It
// runs before validation: the rows of a valid offset array are disjoint, so
// fewer than cap of them are long, and a count above cap (rows that overlap)
// is written nowhere and reported by the caller.
__global__ void k_long_rows(int64_t n, int64_t nnz, const int64_t* __restrict__ rp, int32_t* __restrict__ rows,
                            int64_t* __restrict__ len, unsigned long long cap,
                            unsigned long long* __restrict__ count) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = rp[u], e = rp[u + 1];
        if (b < 0 || e < b || e > nnz || !is_long_row(b, e)) continue;
        const unsigned long long i = atomicAdd(count, 1ull);
        if (i >= cap) continue;
        rows[i] = (int32_t)u;
        len[i] = e - b;
    }
}

// segment s of the long rows: row index i (seg_off[i] <= s < seg_off[i+1])
// and the entry range [pb, pe)
__device__ __forceinline__ void long_segment(int64_t s, const int32_t* __restrict__ rows,
                                             const int64_t* __restrict__ seg_off, int64_t count,
                                             const int64_t* __restrict__ rp, int64_t& u, int64_t& b, int64_t& pb,
                                             int64_t& pe) {
    int64_t lo = 0, hi = count;  // last i with seg_off[i] <= s
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (seg_off[mid] <= s) lo = mid; else hi = mid;
    }
    u = rows[lo];
    b = rp[u];
    const int64_t e = rp[u + 1];
    pb = b + (s - seg_off[lo]) * kLongSeg;
    pe = min(pb + kLongSeg, e);
}

// the two fingerprint sums of a warp's lanes, added to fp_out[0..1]
__device__ __forceinline__ void fp_flush(unsigned long long (&fp)[2], unsigned long long* fp_out) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fp[0] += __shfl_xor_sync(kFull, fp[0], o);
        fp[1] += __shfl_xor_sync(kFull, fp[1], o);
    }
    if ((threadIdx.x & 31) == 0 && (fp[0] | fp[1])) {
        atomicAdd(fp_out, fp[0]);
        atomicAdd(fp_out + 1, fp[1]);
    }
}

template <bool BY_LENGTH, bool FP = false>
__global__ void k_validate_split(int per, int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                 const int32_t* __restrict__ col, int32_t* __restrict__ nlow,
                                 int64_t* __restrict__ upcnt, int* __restrict__ err,
                                 unsigned long long* __restrict__ searched, uint32_t* __restrict__ mirror,
                                 unsigned long long* __restrict__ fp_out) {
    __shared__ uint32_t pre[kThreads / 32][row_pool::kWords];
    __shared__ int64_t begin[kThreads / 32][32];
    __shared__ int lows[kThreads / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long fp[2] = {0ull, 0ull};
    int found = 0;
    bool bad_entry = false;
    const int64_t groups = (n + per - 1) / per;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t u0 = per * g, mine = lane < per ? u0 + lane : n;
        int64_t b = 0;
        int len = 0;
        if (mine < n) {
            b = rp[mine];
            const int64_t e = rp[mine + 1];
            if (b < 0 || e < b || e > nnz || (mine == 0 && b != 0) || (mine == n - 1 && e != nnz)) {
                atomicOr(err, 1);
            } else if (is_long_row(b, e)) {  // counted by k_validate_long
                // a graph of at most kLongRow vertices: too long to be simple
                if (n <= kLongRow) atomicOr(err, 2);
            } else if (e - b <= kPoolRow) {
                len = (int)(e - b);
            }
        }
        begin[w][lane] = b;
        lows[w][lane] = 0;
        row_pool pool(pre[w], len);
        for (int e0 = 0; e0 < pool.total; e0 += 32) {
            const int x = e0 + lane;
            const auto [r, at, same] = pool.block(e0);
            bool low = false;
            if (x < pool.total) {
                const int64_t rb = begin[w][r], p = rb + (x - at), re = rb + pool.length(r);
                if (!validate_entry<BY_LENGTH, FP>(n, nnz, rp, col, u0 + r, rb, re, p, mirror, low, found, fp))
                    bad_entry = true;
            }
            const unsigned m = __ballot_sync(kFull, low) & same;
            if (lane == __ffs(same) - 1) lows[w][r] += __popc(m);
            __syncwarp();
        }
        if (mine < n && len > 0) {  // the others are zeroed beforehand, and may have been counted since
            nlow[mine] = lows[w][lane];
            upcnt[mine] = len - lows[w][lane];
        }
    }
    spread_rows(
        n,
        [&](int64_t u) {
            const int64_t b = rp[u], e = rp[u + 1];
            return b >= 0 && e <= nnz && e - b > kPoolRow && !is_long_row(b, e);
        },
        [&](int64_t u) {
            const int64_t b = rp[u], e = rp[u + 1];
            int low = 0, in_row = 0;
            bool bad = false;
            validate_entries<BY_LENGTH, FP>(n, nnz, rp, col, u, b, e, b, e, mirror, low, in_row, bad, fp);
            if (lane == 0) {
                found += in_row;
                nlow[u] = low;
                upcnt[u] = (e - b) - low;
            }
            bad_entry |= bad;
        });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) found += __shfl_xor_sync(kFull, found, o);
    if (lane == 0 && found) atomicAdd(searched, (unsigned long long)found);
    if (bad_entry) atomicOr(err, 2);
    if constexpr (FP) fp_flush(fp, fp_out);
}

// the long rows, one warp per segment; the counts add up per row
template <bool BY_LENGTH, bool FP = false>
__global__ void k_validate_long(int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                const int32_t* __restrict__ col, const int32_t* __restrict__ rows,
                                const int64_t* __restrict__ seg_off, int64_t count, int64_t segs,
                                int32_t* __restrict__ nlow, int64_t* __restrict__ upcnt, int* __restrict__ err,
                                unsigned long long* __restrict__ searched, uint32_t* __restrict__ mirror,
                                unsigned long long* __restrict__ fp_out) {
    const int lane = threadIdx.x & 31;
    unsigned long long fp[2] = {0ull, 0ull};
    for (int64_t sg = warp_id_global(); sg < segs; sg += warp_count_global()) {
        int64_t u, b, pb, pe;
        long_segment(sg, rows, seg_off, count, rp, u, b, pb, pe);
        int low = 0, found = 0;
        bool rowbad = false;
        validate_entries<BY_LENGTH, FP>(n, nnz, rp, col, u, b, rp[u + 1], pb, pe, mirror, low, found, rowbad, fp);
        if (lane == 0) {
            atomicAdd(nlow + u, low);
            atomicAdd(reinterpret_cast<unsigned long long*>(upcnt + u), (unsigned long long)((pe - pb) - low));
            if (found) atomicAdd(searched, (unsigned long long)found);
            if (rowbad) atomicOr(err, 2);
        }
    }
    if constexpr (FP) fp_flush(fp, fp_out);
}

// ---- (1,2): vertices relabelled by degree class ----------------------------
// The k-core pass gathers tau at the neighbour ids of every row.  With ids in
// no particular order (a scrambled R-MAT), the gathers of a large graph go to
// DRAM; most of them hit the few high-degree vertices, but those are spread
// over the whole tau array, one value per line.  The build therefore gives
// the vertices new ids by degree class, floor(log2 d) descending, stable
// within a class, so that the values most gathered share lines.  Results
// are permuted back at the boundary (nd_api.cu).
constexpr int kClasses = 34;         // 0..31 by degree, 32: degree 0, 33: past n
constexpr int kRelabelTile = 4096;   // vertices per block (16 rounds of 256)

__device__ __forceinline__ int degree_class(int64_t d) {
    return d == 0 ? 32 : 31 - (63 - __clzll((unsigned long long)d));  // high degree first
}

__global__ void k_class_count(int64_t n, const int64_t* __restrict__ rp, int64_t* __restrict__ cnt,
                              int64_t nblocks) {
    __shared__ unsigned c[kClasses];
    for (int i = threadIdx.x; i < kClasses; i += blockDim.x) c[i] = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * kRelabelTile;
    for (int64_t v = t0 + threadIdx.x; v < min(t0 + kRelabelTile, n); v += blockDim.x)
        atomicAdd(&c[degree_class(rp[v + 1] - rp[v])], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < kClasses - 1; i += blockDim.x) cnt[(int64_t)i * nblocks + blockIdx.x] = c[i];
}

// new id = start of (class, block) + earlier vertices of the class in the block
__global__ void k_class_scatter(int64_t n, const int64_t* __restrict__ rp, const int64_t* __restrict__ off,
                                int64_t nblocks, int32_t* __restrict__ to_new, int32_t* __restrict__ to_old) {
    __shared__ unsigned wcnt[kThreads / 32][kClasses];
    __shared__ unsigned run[kClasses];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kClasses; i += blockDim.x) run[i] = 0;
    const int64_t t0 = (int64_t)blockIdx.x * kRelabelTile;
    for (int64_t r0 = t0; r0 < t0 + kRelabelTile; r0 += kThreads) {
        const int64_t v = r0 + threadIdx.x;
        const bool ok = v < n && v < t0 + kRelabelTile;
        const int k = ok ? degree_class(rp[v + 1] - rp[v]) : kClasses - 1;
        for (int i = lane; i < kClasses; i += 32) wcnt[warp][i] = 0;
        __syncthreads();
        const unsigned same = __match_any_sync(0xffffffffu, k);
        const unsigned rank = __popc(same & ((1u << lane) - 1u));
        if (rank == 0) wcnt[warp][k] = __popc(same);
        __syncthreads();
        if (ok) {
            unsigned before = run[k];
            for (int w = 0; w < warp; ++w) before += wcnt[w][k];
            const int64_t id = off[(int64_t)k * nblocks + blockIdx.x] + before + rank;
            to_new[v] = (int32_t)id;
            to_old[id] = (int32_t)v;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kClasses; i += blockDim.x) {
            unsigned tot = 0;
            for (int w = 0; w < kThreads / 32; ++w) tot += wcnt[w][i];
            run[i] += tot;
        }
        __syncthreads();
    }
}

__global__ void k_new_degrees(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ to_new,
                              int64_t* __restrict__ len) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        len[to_new[v]] = rp[v + 1] - rp[v];
}

// The rows under the new ids are ordered by the octave of the id,
// floor(log2 id): ids ascend by degree class, so the neighbours of large tau
// come first.  A pass then finds tau(R) entries at or above tau(R) early, and
// knows from the octave that no later entry can reach a value (h->oct_max).
// R-MAT scale 20 on the CPU: a converged pass reads 0.6 of the entries, 0.92
// in the caller's order; sorting fully by degree gains no more.
__device__ __forceinline__ int octave_of(uint32_t id) { return 31 - __clz(id | 1u); }

constexpr int kSortRow = 512;  // entries of a row that one warp orders in shared memory

// How a row is ordered: the key of the entry at CSR position p, its bucket
// (0..31, the order of the row), where row u's output begins, and the write.
struct NewIdOrder {  // k-core relabelling: new ids, by octave
    const int32_t* __restrict__ col;
    const int32_t* __restrict__ to_new;
    const int64_t* __restrict__ nrp;
    int32_t* __restrict__ ncol;
    __device__ __forceinline__ uint32_t key(int64_t p) const { return (uint32_t)to_new[col[p]]; }
    static __device__ __forceinline__ int bucket(uint32_t key) { return octave_of(key); }
    __device__ __forceinline__ int64_t begin(int64_t u, int64_t) const { return nrp[to_new[u]]; }
    __device__ __forceinline__ void write(int64_t at, int64_t, uint32_t key) const { ncol[at] = (int32_t)key; }
};
struct DegreeOrder {  // no-storage passes: the caller's ids with their slots, by degree class, high first
    const int64_t* __restrict__ rp;
    const int32_t* __restrict__ col;
    int32_t* __restrict__ vertex;
    uint32_t* __restrict__ slot;
    __device__ __forceinline__ uint32_t key(int64_t p) const {
        const int32_t v = col[p];
        return (uint32_t)degree_class(rp[v + 1] - rp[v]);  // a neighbour has a neighbour: below 32
    }
    static __device__ __forceinline__ int bucket(uint32_t key) { return (int)key; }
    __device__ __forceinline__ int64_t begin(int64_t, int64_t b) const { return b; }
    __device__ __forceinline__ void write(int64_t at, int64_t p, uint32_t) const {
        vertex[at] = col[p];
        slot[at] = (uint32_t)p;
    }
};

// rows of up to kSortRow entries: up to 8 are ranked across eight lanes, up to
// 32 across the warp; longer rows go through 32 shared counters, one warp each
template <typename K>
__global__ void __launch_bounds__(kThreads) k_order_rows(int per, int64_t n, const int64_t* __restrict__ rp, K k) {
    __shared__ uint32_t stage[kThreads / 32][kSortRow];
    __shared__ uint32_t cur[kThreads / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t groups = (n + per - 1) / per;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t u0 = per * g, mine = lane < per ? u0 + lane : n;
        const int64_t b = mine < n ? rp[mine] : 0, d = mine < n ? rp[mine + 1] - b : 0;
        const int64_t out = d > 0 && d <= 32 ? k.begin(mine, b) : 0;
        if (d == 1) k.write(out, b, k.key(b));
        for (unsigned todo = __ballot_sync(kFull, d >= 2 && d <= 8); todo;) {
            int r = -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int f = todo ? __ffs(todo) - 1 : -1;
                if (lane / 8 == q) r = f;
                todo &= todo - 1;  // 0 stays 0
            }
            const int64_t rb = __shfl_sync(kFull, b, max(r, 0)), ro = __shfl_sync(kFull, out, max(r, 0));
            const int64_t any_d = __shfl_sync(kFull, d, max(r, 0));
            const int j = lane & 7, rd = r >= 0 ? (int)any_d : 0;
            const uint32_t key = j < rd ? k.key(rb + j) : 0xffffffffu;
            int rank = 0;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const uint32_t x = __shfl_sync(kFull, key, o, 8);
                rank += x < key || (x == key && o < j);
            }
            if (j < rd) k.write(ro + rank, rb + j, key);
        }
        for (unsigned todo = __ballot_sync(kFull, d > 8 && d <= 32); todo; todo &= todo - 1) {
            const int r = __ffs(todo) - 1;
            const int64_t rb = __shfl_sync(kFull, b, r), ro = __shfl_sync(kFull, out, r);
            const int rd = (int)__shfl_sync(kFull, d, r);
            const uint32_t key = lane < rd ? k.key(rb + lane) : 0xffffffffu;
            int rank = 0;
            for (int o = 0; o < rd; ++o) {
                const uint32_t x = __shfl_sync(kFull, key, o);
                rank += x < key || (x == key && o < lane);
            }
            if (lane < rd) k.write(ro + rank, rb + lane, key);
        }
    }
    spread_rows(
        n,
        [&](int64_t u) {
            const int64_t d = rp[u + 1] - rp[u];
            return d > 32 && d <= kSortRow;  // longer: k_sort_count, k_sort_scatter
        },
        [&](int64_t u) {
            const int64_t b = rp[u], out = k.begin(u, b);
            const int d = (int)(rp[u + 1] - b);
            cur[w][lane] = 0;
            __syncwarp();
            for (int j = lane; j < d; j += 32) {
                const uint32_t key = k.key(b + j);
                stage[w][j] = key;
                atomicAdd(&cur[w][K::bucket(key)], 1u);
            }
            __syncwarp();
            const uint32_t c = cur[w][lane];
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            cur[w][lane] = incl - c;
            __syncwarp();
            for (int j = lane; j < d; j += 32) {
                const uint32_t key = stage[w][j];
                k.write(out + atomicAdd(&cur[w][K::bucket(key)], 1u), b + j, key);
            }
            __syncwarp();
        });
}

// the rows longer than kSortRow and the number of their kLongSeg segments
__global__ void k_sort_list(int64_t n, const int64_t* __restrict__ rp, int32_t* __restrict__ rows,
                            int64_t* __restrict__ segs, unsigned long long* __restrict__ count) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = rp[u + 1] - rp[u];
        if (d <= kSortRow) continue;
        const unsigned long long i = atomicAdd(count, 1ull);
        rows[i] = (int32_t)u;
        segs[i] = (d + kLongSeg - 1) / kLongSeg;
    }
}

// segment sg of the listed rows (seg_off: scanned segment counts): its row
// and entries, and where its 32 counters lie: cells[cell + octave * stride],
// a row's cells octave by octave, so that their scan gives every segment its
// first slot per octave
struct sort_segment {
    int64_t u, b, pb, pe, row_cell, cell, stride;
    __device__ __forceinline__ sort_segment(int64_t sg, const int32_t* __restrict__ rows,
                                            const int64_t* __restrict__ seg_off, int64_t count,
                                            const int64_t* __restrict__ rp) {
        int64_t lo = 0, hi = count;  // last i with seg_off[i] <= sg
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (seg_off[mid] <= sg) lo = mid; else hi = mid;
        }
        u = rows[lo];
        b = rp[u];
        const int64_t s = sg - seg_off[lo];
        pb = b + s * kLongSeg;
        pe = min(pb + kLongSeg, rp[u + 1]);
        row_cell = 32 * seg_off[lo];
        stride = seg_off[lo + 1] - seg_off[lo];
        cell = row_cell + s;
    }
};

template <typename K>
__global__ void __launch_bounds__(kThreads) k_sort_count(const int64_t* __restrict__ rp, K k,
                                                         const int32_t* __restrict__ rows,
                                                         const int64_t* __restrict__ seg_off, int64_t count,
                                                         int64_t segs, int64_t* __restrict__ cells) {
    __shared__ uint32_t cnt[kThreads / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t sg = warp_id_global(); sg < segs; sg += warp_count_global()) {
        const sort_segment x(sg, rows, seg_off, count, rp);
        cnt[w][lane] = 0;
        __syncwarp();
        for (int64_t p = x.pb + lane; p < x.pe; p += 32) atomicAdd(&cnt[w][K::bucket(k.key(p))], 1u);
        __syncwarp();
        cells[x.cell + lane * x.stride] = cnt[w][lane];
        __syncwarp();
    }
}

template <typename K>
__global__ void __launch_bounds__(kThreads) k_sort_scatter(const int64_t* __restrict__ rp, K k,
                                                           const int32_t* __restrict__ rows,
                                                           const int64_t* __restrict__ seg_off, int64_t count,
                                                           int64_t segs, const int64_t* __restrict__ cells) {
    __shared__ uint32_t cur[kThreads / 32][32];  // a row has fewer than 2^31 entries
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t sg = warp_id_global(); sg < segs; sg += warp_count_global()) {
        const sort_segment x(sg, rows, seg_off, count, rp);
        cur[w][lane] = (uint32_t)(cells[x.cell + lane * x.stride] - cells[x.row_cell]);
        __syncwarp();
        const int64_t out = k.begin(x.u, x.b);
        for (int64_t p = x.pb + lane; p < x.pe; p += 32) {
            const uint32_t key = k.key(p);
            k.write(out + atomicAdd(&cur[w][K::bucket(key)], 1u), p, key);
        }
        __syncwarp();
    }
}

__global__ void k_permute_i32(int64_t n, const int32_t* __restrict__ idx, const int32_t* __restrict__ in,
                              int32_t* __restrict__ out, int scatter) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (scatter) out[idx[i]] = in[i];
        else out[i] = in[idx[i]];
    }
}

// (2,3) relabelling: the key (new u, new v) of every entry, at its own
// position (the sort that follows fixes the order)
__device__ __forceinline__ void relabel_key_entries(const int32_t* __restrict__ col, const int32_t* __restrict__ to_new,
                                                    int bits, unsigned long long* __restrict__ keys, int64_t u,
                                                    int64_t pb, int64_t pe) {
    const unsigned long long hi = (unsigned long long)to_new[u] << bits;
    for (int64_t p = pb + (threadIdx.x & 31); p < pe; p += 32) keys[p] = hi | (unsigned long long)to_new[col[p]];
}

__global__ void k_relabel_keys(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                               const int32_t* __restrict__ to_new, int bits, unsigned long long* __restrict__ keys) {
    for (int64_t u = warp_id_global(); u < n; u += warp_count_global()) {
        const int64_t b = rp[u], e = rp[u + 1];
        if (is_long_row(b, e)) continue;  // k_relabel_keys_long
        relabel_key_entries(col, to_new, bits, keys, u, b, e);
    }
}

__global__ void k_relabel_keys_long(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                    const int32_t* __restrict__ to_new, int bits, unsigned long long* __restrict__ keys,
                                    const int32_t* __restrict__ rows, const int64_t* __restrict__ seg_off,
                                    int64_t count, int64_t segs) {
    for (int64_t sg = warp_id_global(); sg < segs; sg += warp_count_global()) {
        int64_t u, b, pb, pe;
        long_segment(sg, rows, seg_off, count, rp, u, b, pb, pe);
        relabel_key_entries(col, to_new, bits, keys, u, pb, pe);
    }
}

__global__ void k_keys_to_col(int64_t nnz, const unsigned long long* __restrict__ keys, int bits,
                              int32_t* __restrict__ col) {
    const unsigned long long mask = (1ull << bits) - 1ull;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nnz; j += (int64_t)gridDim.x * blockDim.x)
        col[j] = (int32_t)(keys[j] & mask);
}

// new edge e = (e_u[e], e_v[e]) -> the caller's edge id: its endpoints in
// caller ids, smaller first, and the rank of the larger among the smaller
// one's larger neighbours in the caller's CSR
__global__ void k_edge_map(int64_t m, const int32_t* __restrict__ e_u, const int32_t* __restrict__ e_v,
                           const int32_t* __restrict__ vto_old, const int64_t* __restrict__ c_rp,
                           const int32_t* __restrict__ c_col, const int32_t* __restrict__ c_nlow,
                           const int64_t* __restrict__ c_up, int32_t* __restrict__ to_new,
                           int32_t* __restrict__ to_old, int* __restrict__ err) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = vto_old[e_u[e]], b = vto_old[e_v[e]];
        const int32_t x = a < b ? a : b, y = a < b ? b : a;
        const int64_t first = c_rp[x] + c_nlow[x], end = c_rp[x + 1];
        const int64_t pos = lower_bound_i32(c_col, first, end, y);
        if (pos >= end || c_col[pos] != y) { atomicOr(err, 1); continue; }
        const int64_t cid = c_up[x] + (pos - first);
        to_old[e] = (int32_t)cid;
        to_new[cid] = (int32_t)e;
    }
}

// r-clique tuples of a relabelled (2,3) handle: caller vertex ids, at the
// caller's edge ids
__global__ void k_r_cliques_mapped(int64_t N, const int32_t* __restrict__ e_u, const int32_t* __restrict__ e_v,
                                   const int32_t* __restrict__ vto_old, const int32_t* __restrict__ to_old,
                                   int32_t* __restrict__ out) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = vto_old[e_u[e]], b = vto_old[e_v[e]];
        const int64_t c = to_old[e];
        out[2 * c] = a < b ? a : b;
        out[2 * c + 1] = a < b ? b : a;
    }
}

// ---- canonical edge ids (one warp per vertex) ------------------------------
// Edge (u,v), u < v, gets id up_start[u] + (rank of v among u's larger
// neighbours): lexicographic order.  eid[p] is the id of the edge at CSR
// position p, for both directions (the reverse entry comes from mirror,
// written by the validation, when there is one).  For the (2,3) adjacency
// layout it also writes, per edge (x,y) with x < y, e_pos = (P(x,y), P(y,x)).
__device__ __forceinline__ void edge_id_entries(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                const int32_t* __restrict__ nlow,
                                                const int64_t* __restrict__ up_start, uint32_t* __restrict__ eid,
                                                int32_t* __restrict__ e_u, int32_t* __restrict__ e_v,
                                                const uint32_t* __restrict__ mirror, uint2* __restrict__ e_pos,
                                                int64_t u, int64_t b, int64_t pb, int64_t pe) {
    const int lane = threadIdx.x & 31;
    const int64_t first_up = b + nlow[u];
    const int64_t base = up_start[u];
    for (int64_t p = pb + lane; p < pe; p += 32) {
        int32_t v = col[p];
        if (p >= first_up) {
            int64_t id = base + (p - first_up);
            eid[p] = (uint32_t)id;
            e_u[id] = (int32_t)u;
            e_v[id] = v;
        } else {
            const int64_t vfirst = rp[v] + nlow[v];
            // the reverse entry: recorded by the validation when available
            const int64_t pos = mirror ? (int64_t)mirror[p]
                                       : lower_bound_i32(col, vfirst, rp[v + 1], (int32_t)u);
            const int64_t id = up_start[v] + (pos - vfirst);
            eid[p] = (uint32_t)id;
            // edge (v,u), v < u: entry pos = P(v,u), entry p = P(u,v)
            if (e_pos) e_pos[id] = make_uint2((uint32_t)pos, (uint32_t)p);
        }
    }
}

__global__ void k_edge_ids(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                           const int32_t* __restrict__ nlow, const int64_t* __restrict__ up_start,
                           uint32_t* __restrict__ eid, int32_t* __restrict__ e_u,
                           int32_t* __restrict__ e_v, const uint32_t* __restrict__ mirror,
                           uint2* __restrict__ e_pos) {
    for (int64_t u = warp_id_global(); u < n; u += warp_count_global()) {
        const int64_t b = rp[u], e = rp[u + 1];
        if (is_long_row(b, e)) continue;  // k_edge_ids_long
        edge_id_entries(rp, col, nlow, up_start, eid, e_u, e_v, mirror, e_pos, u, b, b, e);
    }
}

__global__ void k_edge_ids_long(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                const int32_t* __restrict__ nlow, const int64_t* __restrict__ up_start,
                                uint32_t* __restrict__ eid, int32_t* __restrict__ e_u, int32_t* __restrict__ e_v,
                                const uint32_t* __restrict__ mirror, uint2* __restrict__ e_pos,
                                const int32_t* __restrict__ rows, const int64_t* __restrict__ seg_off,
                                int64_t count, int64_t segs) {
    for (int64_t sg = warp_id_global(); sg < segs; sg += warp_count_global()) {
        int64_t u, b, pb, pe;
        long_segment(sg, rows, seg_off, count, rp, u, b, pb, pe);
        edge_id_entries(rp, col, nlow, up_start, eid, e_u, e_v, mirror, e_pos, u, b, pb, pe);
    }
}

// ---- (2,3): triangles by degree orientation --------------------------------
// Vertex u precedes v iff (d_u, u) < (d_v, v).  Orienting every edge from the
// earlier to the later endpoint, each triangle {u,v,w} (u before v before w)
// is found exactly once, as w in out(u) /\ out(v) for the oriented edge
// u -> v; out-lists are at most sqrt(2m) long.  The triangle then adds one
// incidence to each of its three edges, at slots taken from per-edge counters
// (count pass) and cursors (fill pass).  Row order inside an edge's incidence
// row is therefore unspecified; the h-index of a row does not depend on it.
__device__ __forceinline__ bool precedes(int64_t du, int32_t u, int64_t dv, int32_t v) {
    return du < dv || (du == dv && u < v);
}

// count / list the out-neighbours of every vertex in id order, 32 vertices per
// warp (with out_pm: also the CSR positions of the entry and of its reverse)
template <bool FILL>
__global__ void __launch_bounds__(kThreads) k_orient(int per, int64_t n, const int64_t* __restrict__ rp,
                                                     const int32_t* __restrict__ col,
                                                     const uint32_t* __restrict__ eid, int64_t* __restrict__ out_ptr,
                                                     int32_t* __restrict__ out_col, uint32_t* __restrict__ out_eid,
                                                     int32_t* __restrict__ out_src,
                                                     const uint32_t* __restrict__ mirror,
                                                     uint2* __restrict__ out_pm) {
    __shared__ uint32_t pre[kThreads / 32][row_pool::kWords];
    __shared__ int64_t begin[kThreads / 32][32], slots[kThreads / 32][32];  // slots: next output slot of each row
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto put = [&](int64_t slot, int32_t u, int32_t v, int64_t p) {
        out_col[slot] = v;
        out_eid[slot] = __ldg(eid + p);
        out_src[slot] = u;
        if (out_pm) out_pm[slot] = make_uint2((uint32_t)p, __ldg(mirror + p));
    };
    const int64_t groups = (n + per - 1) / per;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t u0 = per * g, mine = lane < per ? u0 + lane : n;
        const int64_t b = mine < n ? rp[mine] : 0, len = mine < n ? rp[mine + 1] - b : 0;
        __syncwarp();
        begin[w][lane] = b;
        slots[w][lane] = FILL && mine < n ? out_ptr[mine] : 0;
        row_pool pool(pre[w], len > kPoolRow ? 0 : (int)len);
        auto entry = [&](bool ok, int r, unsigned same, int64_t p, int64_t du) {
            bool keep = false;
            int32_t v = 0;
            if (ok) {
                v = __ldg(col + p);
                keep = precedes(du, (int32_t)(u0 + r), __ldg(rp + v + 1) - __ldg(rp + v), v);
            }
            const unsigned m = __ballot_sync(kFull, keep) & same;
            const int64_t first = slots[w][r];
            __syncwarp();
            if (lane == __ffs(same) - 1) slots[w][r] = first + __popc(m);
            if (FILL && keep) put(first + __popc(m & lanemask_lt()), (int32_t)(u0 + r), v, p);
            __syncwarp();
        };
        for (int e0 = 0; e0 < pool.total; e0 += 32) {
            const int x = e0 + lane;
            const auto [r, at, same] = pool.block(e0);
            entry(x < pool.total, r, same, begin[w][r] + (x - at), pool.length(r));
        }
        if (!FILL && mine < n && len <= kPoolRow) out_ptr[mine] = slots[w][lane];
    }
    spread_rows(
        n, [&](int64_t u) { return rp[u + 1] - rp[u] > kPoolRow; },
        [&](int64_t u) {
            const int64_t b = rp[u], e = rp[u + 1], du = e - b;
            int64_t slot = FILL ? out_ptr[u] : 0;
            for (int64_t p0 = b; p0 < e; p0 += 32) {
                const int64_t p = p0 + lane;
                bool keep = false;
                int32_t v = 0;
                if (p < e) {
                    v = __ldg(col + p);
                    keep = precedes(du, (int32_t)u, __ldg(rp + v + 1) - __ldg(rp + v), v);
                }
                const unsigned m = __ballot_sync(kFull, keep);
                if (FILL && keep) put(slot + __popc(m & lanemask_lt()), (int32_t)u, v, p);
                slot += __popc(m);
            }
            if (!FILL && lane == 0) out_ptr[u] = slot;
        });
}

#ifndef ND_TRI_COUNT_MIN_BLOCKS
#define ND_TRI_COUNT_MIN_BLOCKS 8  // the count pass (with its records) at full occupancy
#endif
#ifndef ND_TRI_MIN_BLOCKS
#define ND_TRI_MIN_BLOCKS 6  // resident blocks per SM for the searching fill (used when the records do not fit)
#endif
// The searching fill (small builds, and where the records do not fit): one
// warp per oriented edge u -> v, the triangles {u, v, w}, w in out(u) /\
// out(v); the lanes walk the shorter list and search the longer.  The entries
// are CSR positions, each pair ordered by its edge's canonical endpoints (the
// entry of the smaller endpoint first).
// Records (the count pass's, for the fill from records): every triangle found
// from edge k, as the offsets of w in the shorter and in the longer out-list
// (16 bits each: an out-list holds at most sqrt(2m) < 65536 entries, since
// each of its vertices has at least the owner's degree and nnz < 2^32), at
// rec[rec_ptr[k] + i]; rec_ptr[k] reserves min(|out(u)|, |out(v)|) slots, the
// most edge k can find.  rec_cnt[k] = triangles found.
template <typename C>
__global__ void __launch_bounds__(kThreads, ND_TRI_MIN_BLOCKS)
    k_tri_fill_search(int64_t m, const int64_t* __restrict__ out_ptr, const int32_t* __restrict__ out_col,
                      const uint32_t* __restrict__ out_eid, const int32_t* __restrict__ out_src,
                      const uint2* __restrict__ out_pm, C* __restrict__ ctr, uint2* __restrict__ inc) {
    const int lane = threadIdx.x & 31;
    for (int64_t k = warp_id_global(); k < m; k += warp_count_global()) {
        const int32_t u = out_src[k], v = out_col[k];
        const uint32_t e_uv = out_eid[k];
        const uint2 uv = __ldg(out_pm + k);  // P(u,v), P(v,u)
        int64_t ab = out_ptr[u], ae = out_ptr[u + 1], bb = out_ptr[v], be = out_ptr[v + 1];
        bool a_is_u = true;
        if (ae - ab > be - bb) {
            int64_t t = ab; ab = bb; bb = t; t = ae; ae = be; be = t;
            a_is_u = false;
        }
        int64_t lo = bb;
        for (int64_t base = ab; base < ae; base += 32) {
            const int64_t p = base + lane;
            bool found = false;
            int64_t pb = 0;
            int32_t x = 0;
            // the values at p are loaded with x, ahead of the search
            // (coalesced), so only the loads at pb wait for it
            uint32_t ea = 0;
            uint2 pa = make_uint2(0, 0);
            if (p < ae) {
                x = __ldg(out_col + p);
                ea = __ldg(out_eid + p);
                pa = __ldg(out_pm + p);
                pb = lo + nd_lower_bound_n(out_col + lo, (int)(be - lo), x);
                found = (pb < be) && (__ldg(out_col + pb) == x);
            }
            const unsigned bal = __ballot_sync(kFull, found);
            const int nf = __popc(bal);
            if (nf) {
                uint32_t eb = 0;
                uint2 pq = make_uint2(0, 0);
                if (found) {
                    eb = __ldg(out_eid + pb);
                    pq = __ldg(out_pm + pb);
                }
                const uint32_t e_uw = a_is_u ? ea : eb, e_vw = a_is_u ? eb : ea;
                // the three slot reservations are independent: issue them together
                C s0 = 0, s_uw = 0, s_vw = 0;
                if (lane == 0) s0 = atomicAdd(ctr + e_uv, (C)nf);
                if (found) {
                    s_uw = atomicAdd(ctr + e_uw, (C)1);
                    s_vw = atomicAdd(ctr + e_vw, (C)1);
                }
                s0 = __shfl_sync(kFull, s0, 0);
                if (found) {
                    // third vertex w = x; positions P(.,.) of the six entries
                    const uint2 uw = a_is_u ? pa : pq, vw = a_is_u ? pq : pa;  // P(u,w), P(w,u); P(v,w), P(w,v)
                    inc[s0 + __popc(bal & lanemask_lt())] = u < v ? make_uint2(uw.x, vw.x) : make_uint2(vw.x, uw.x);
                    inc[s_uw] = u < x ? make_uint2(uv.x, vw.y) : make_uint2(vw.y, uv.x);
                    inc[s_vw] = v < x ? make_uint2(uv.y, uw.y) : make_uint2(uw.y, uv.y);
                }
            }
            const int64_t last_pb = __shfl_sync(kFull, pb, 31);
            if (base + 32 <= ae) lo = last_pb;
        }
    }
}

// The count: 32 consecutive oriented edges per warp.  The elements of an
// edge's shorter out-list, in whole blocks of 32, are looked up in the longer
// one by the warp; the rests of all 32 edges are then walked as one sequence.
template <bool REC>
__global__ void __launch_bounds__(kThreads, ND_TRI_COUNT_MIN_BLOCKS)
    k_tri_count(int per, int64_t m, const int64_t* __restrict__ out_ptr, const int32_t* __restrict__ out_col,
                const uint32_t* __restrict__ out_eid, const int32_t* __restrict__ out_src, unsigned* __restrict__ ctr,
                const int64_t* __restrict__ rec_ptr, uint32_t* __restrict__ rec, uint32_t* __restrict__ rec_cnt) {
    __shared__ uint32_t pre[kThreads / 32][row_pool::kWords];
    __shared__ uint32_t ab[kThreads / 32][32], bb[kThreads / 32][32], bn[kThreads / 32][32], an[kThreads / 32][32];
    __shared__ uint32_t nf[kThreads / 32][32];  // triangles found from each edge so far
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t groups = (m + per - 1) / per;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t k0 = per * g, mine = lane < per ? k0 + lane : m;
        uint32_t a = 0, b = 0;
        int na = 0, nb = 0;  // out-lists have fewer than 65,536 entries
        if (mine < m) {
            const int32_t u = out_src[mine], v = out_col[mine];
            const int64_t ub = out_ptr[u], ue = out_ptr[u + 1], vb = out_ptr[v], ve = out_ptr[v + 1];
            const bool us = ue - ub <= ve - vb;
            a = (uint32_t)(us ? ub : vb);
            b = (uint32_t)(us ? vb : ub);
            na = (int)(us ? ue - ub : ve - vb);
            nb = (int)(us ? ve - vb : ue - ub);
        }
        __syncwarp();
        ab[w][lane] = a;
        bb[w][lane] = b;
        an[w][lane] = (uint32_t)na;
        bn[w][lane] = (uint32_t)nb;
        nf[w][lane] = 0;
        row_pool pool(pre[w], na & 31);
        // element j of edge r's shorter list
        auto element = [&](bool ok, int r, unsigned same, int j) {
            bool found = false;
            uint32_t p = 0, pb = 0;
            if (ok) {
                p = ab[w][r] + j;
                const uint32_t lb = bb[w][r];
                const int32_t x = __ldg(out_col + p);
                const int at = nd_lower_bound_n(out_col + lb, (int)bn[w][r], x);
                pb = lb + at;
                found = at < (int)bn[w][r] && __ldg(out_col + pb) == x;
            }
            const unsigned all = __ballot_sync(kFull, found);
            if (!all) return;
            const unsigned hit = all & same;
            const uint32_t before = nf[w][r];
            __syncwarp();
            if (lane == __ffs(same) - 1 && hit) nf[w][r] = before + __popc(hit);
            if (found) {
                atomicAdd(ctr + __ldg(out_eid + p), 1u);
                atomicAdd(ctr + __ldg(out_eid + pb), 1u);
                if (REC)
                    rec[rec_ptr[k0 + r] + before + __popc(hit & lanemask_lt())] =
                        (uint32_t)j | ((pb - bb[w][r]) << 16);
            }
            __syncwarp();
        };
        for (unsigned todo = __ballot_sync(kFull, na >= 32); todo; todo &= todo - 1) {
            const int r = __ffs(todo) - 1, whole = (int)an[w][r] & ~31;
            for (int j = 0; j < whole; j += 32) element(true, r, kFull, j + lane);
        }
        for (int e0 = 0; e0 < pool.total; e0 += 32) {
            const int x = e0 + lane;
            const auto [r, at, same] = pool.block(e0);
            element(x < pool.total, r, same, ((int)an[w][r] & ~31) + x - at);
        }
        if (mine < m) {
            const uint32_t c = nf[w][lane];
            if (c) atomicAdd(ctr + out_eid[mine], c);
            if (REC) rec_cnt[mine] = c;
        }
    }
}

// The fill from the count pass's records: 32 consecutive oriented edges per
// warp, four recorded triangles per lane at a time, so no search is repeated.
// The six positions of a triangle are read at the recorded offsets of w in the
// two out-lists; slots and entries are as in the searching fill.
// Bound by the chain record -> list entries -> slots -> writes and by the L2
// traffic of the slot atomics and scattered 8-byte writes.  Registers for tasks
// in flight are worth more than warps: one task at 5 blocks per SM takes 22.8 ms
// on an R-MAT of 1,048,576 vertices (390M triangles), two at 3 blocks 20.5, at
// 4 blocks 21.5, four at 2 blocks 19.6; 100K vertices 0.833, 0.822, 0.821 and
// 0.833 ms.
#ifndef ND_FILL_TASKS
#define ND_FILL_TASKS 4
#endif
#ifndef ND_FILL_MIN_BLOCKS
#define ND_FILL_MIN_BLOCKS 2
#endif
template <typename C>
__global__ void __launch_bounds__(kThreads, ND_FILL_MIN_BLOCKS)
    k_tri_fill_rec(int per, int64_t m, const int64_t* __restrict__ out_ptr, const int32_t* __restrict__ out_col,
                   const uint32_t* __restrict__ out_eid, const int32_t* __restrict__ out_src,
                   const uint2* __restrict__ out_pm, C* __restrict__ ctr, uint2* __restrict__ inc,
                   const int64_t* __restrict__ rec_ptr, const uint32_t* __restrict__ rec,
                   const uint32_t* __restrict__ rec_cnt) {
    __shared__ uint32_t pre[kThreads / 32][row_pool::kWords];
    __shared__ uint32_t ab[kThreads / 32][32], bb[kThreads / 32][32];
    __shared__ int32_t vu[kThreads / 32][32], vv[kThreads / 32][32];
    __shared__ bool a_is[kThreads / 32][32];  // the shorter list is out(u)
    __shared__ int64_t rp0[kThreads / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t groups = (m + per - 1) / per;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t k0 = per * g, mine = lane < per ? k0 + lane : m;
        const int c = mine < m ? (int)__ldg(rec_cnt + mine) : 0;
        if (!__any_sync(kFull, c > 0)) continue;
        __syncwarp();
        if (c > 0) {
            const int32_t u = out_src[mine], v = out_col[mine];
            const int64_t ub = out_ptr[u], ue = out_ptr[u + 1], vb = out_ptr[v], ve = out_ptr[v + 1];
            const bool us = ue - ub <= ve - vb;  // the same choice of the shorter list as the count pass
            ab[w][lane] = (uint32_t)(us ? ub : vb);
            bb[w][lane] = (uint32_t)(us ? vb : ub);
            vu[w][lane] = u;
            vv[w][lane] = v;
            a_is[w][lane] = us;
            rp0[w][lane] = rec_ptr[mine];
        }
        row_pool pool(pre[w], c);
        constexpr int U = ND_FILL_TASKS;
        for (int e0 = 0; e0 < pool.total; e0 += 32 * U) {
            int r[U];
            unsigned same[U];
            uint32_t p[U], pb[U];
            bool found[U];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const int i = e0 + 32 * t + lane;
                found[t] = i < pool.total;
                const row_pool::place of = pool.block(e0 + 32 * t);
                r[t] = of.row;
                same[t] = of.same;
                p[t] = found[t] ? __ldg(rec + rp0[w][of.row] + (i - of.at)) : 0;
            }
            uint32_t ea[U], eb[U], e_uv[U];
            uint2 pa[U], pq[U], uv[U];
            int32_t x[U];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                if (found[t]) {
                    pb[t] = bb[w][r[t]] + (p[t] >> 16);
                    p[t] = ab[w][r[t]] + (p[t] & 0xffffu);
                    e_uv[t] = __ldg(out_eid + k0 + r[t]);
                    ea[t] = __ldg(out_eid + p[t]);
                    eb[t] = __ldg(out_eid + pb[t]);
                    uv[t] = __ldg(out_pm + k0 + r[t]);
                    x[t] = __ldg(out_col + p[t]);
                    pa[t] = __ldg(out_pm + p[t]);
                    pq[t] = __ldg(out_pm + pb[t]);
                }
            }
            C s0[U], s_uw[U], s_vw[U];
            // the slot reservations are independent: issue them together
#pragma unroll
            for (int t = 0; t < U; ++t) {
                same[t] &= __ballot_sync(kFull, found[t]);
                const bool a_is_u = a_is[w][r[t]];
                s0[t] = 0;
                if (found[t]) {
                    if (lane == __ffs(same[t]) - 1) s0[t] = atomicAdd(ctr + e_uv[t], (C)__popc(same[t]));
                    s_uw[t] = atomicAdd(ctr + (a_is_u ? ea[t] : eb[t]), (C)1);
                    s_vw[t] = atomicAdd(ctr + (a_is_u ? eb[t] : ea[t]), (C)1);
                }
            }
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const bool a_is_u = a_is[w][r[t]];
                const C first = __shfl_sync(kFull, s0[t], found[t] ? __ffs(same[t]) - 1 : lane);
                if (found[t]) {
                    const int32_t u = vu[w][r[t]], v = vv[w][r[t]];
                    const uint2 uw = a_is_u ? pa[t] : pq[t], vw = a_is_u ? pq[t] : pa[t];
                    inc[first + __popc(same[t] & lanemask_lt())] =
                        u < v ? make_uint2(uw.x, vw.x) : make_uint2(vw.x, uw.x);
                    inc[s_uw[t]] = u < x[t] ? make_uint2(uv[t].x, vw.y) : make_uint2(vw.y, uv[t].x);
                    inc[s_vw[t]] = v < x[t] ? make_uint2(uv[t].y, uw.y) : make_uint2(uw.y, uv[t].y);
                }
            }
        }
    }
}

// the record slots of each oriented edge: min(|out(u)|, |out(v)|)
__global__ void k_rec_bound(int64_t m, const int64_t* __restrict__ out_ptr, const int32_t* __restrict__ out_src,
                            const int32_t* __restrict__ out_col, int64_t* __restrict__ rec_ptr) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = out_src[k], v = out_col[k];
        const int64_t a = out_ptr[u + 1] - out_ptr[u], b = out_ptr[v + 1] - out_ptr[v];
        rec_ptr[k] = a < b ? a : b;
    }
}

__global__ void k_widen_u32(int64_t m, const unsigned* __restrict__ in, int64_t* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (int64_t)in[i];
}

__global__ void k_narrow_u32(int64_t m, const int64_t* __restrict__ in, unsigned* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (unsigned)in[i];
}

// ---- (2,3) adjacency layout: order each row by its third vertex -----------
// The entries of the row of edge (x,y) are pairs (P(x,w), P(y,w)) over the
// triangles {x,y,w}, in fill order.  Both components grow with w, so the
// rank of an entry is the rank of its component in the shorter of the two
// adjacency lists, N(s): one bit per position of N(s) marks the row's
// entries, and rank = (bits set in earlier words) + (bits below it in its
// word).  O(d + deg(s)/32) per row, no comparison sort.  Rows up to 32
// entries are ranked by comparing keys across eight lanes or the warp instead.
// A warp takes 32 rows at a time, the longer ones one by one; the bit and prefix
// words sit in shared memory (kRankWords per
// warp); a row whose shorter list needs more words is left to the overflow
// pass, which uses global scratch.
constexpr int kRankWarps = 8;
#ifndef ND_RANK_WORDS
#define ND_RANK_WORDS 512  // 16,384 positions per warp; 32 KB per block
#endif
constexpr int kRankWords = ND_RANK_WORDS;

__device__ __forceinline__ void rank_row(const uint2* __restrict__ src, uint2* __restrict__ dst, int64_t jb,
                                         int64_t d, int comp, uint32_t base, int64_t nw,
                                         uint32_t* __restrict__ bm, uint32_t* __restrict__ pre) {
    const int lane = threadIdx.x & 31;
    for (int64_t w = lane; w < nw; w += 32) bm[w] = 0u;
    __syncwarp();
    for (int64_t j = jb + lane; j < jb + d; j += 32) {
        const uint2 e = src[j];
        const uint32_t k = (comp ? e.y : e.x) - base;
        atomicOr(bm + (k >> 5), 1u << (k & 31));
    }
    __syncwarp();
    uint32_t run = 0;
    for (int64_t w0 = 0; w0 < nw; w0 += 32) {
        const int64_t w = w0 + lane;
        const uint32_t c = w < nw ? (uint32_t)__popc(bm[w]) : 0u;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (w < nw) pre[w] = run + incl - c;
        run += __shfl_sync(kFull, incl, 31);
    }
    __syncwarp();
    for (int64_t j = jb + lane; j < jb + d; j += 32) {
        const uint2 e = src[j];
        const uint32_t k = (comp ? e.y : e.x) - base;
        const uint32_t rank = pre[k >> 5] + (uint32_t)__popc(bm[k >> 5] & ((1u << (k & 31)) - 1u));
        dst[jb + rank] = e;
    }
    __syncwarp();
}

// BIG = false: every row, bits in shared memory; rows that need more than
// kRankWords words are appended to `over` (count in over_ctr[0], largest
// word count in over_ctr[1]).  BIG = true: the rows in `over`, bits in
// global scratch of 2 * scratch_words words per warp.
template <bool BIG>
__global__ void __launch_bounds__(32 * kRankWarps)
k_row_rank(int per, int64_t N, const int64_t* __restrict__ inc_ptr, const int32_t* __restrict__ e_u,
           const int32_t* __restrict__ e_v, const int64_t* __restrict__ rp, const uint2* __restrict__ src,
           uint2* __restrict__ dst, uint32_t* __restrict__ over, unsigned long long* __restrict__ over_ctr,
           uint32_t* __restrict__ scratch, int64_t scratch_words) {
    extern __shared__ uint32_t rank_smem[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    uint32_t *bm, *pre;
    if (BIG) {
        bm = scratch + (size_t)2 * scratch_words * warp_id_global();
        pre = bm + scratch_words;
    } else {
        bm = rank_smem + (size_t)2 * kRankWords * wib;
        pre = bm + kRankWords;
    }
    auto long_row = [&](int64_t R, int64_t jb, int64_t d) {
        const int32_t x = e_u[R], y = e_v[R];
        const int64_t dx = rp[x + 1] - rp[x], dy = rp[y + 1] - rp[y];
        const int comp = dx <= dy ? 0 : 1;
        const uint32_t base = (uint32_t)rp[comp ? y : x];
        const int64_t nw = ((comp ? dy : dx) + 31) / 32;
        if (!BIG && nw > kRankWords) {
            if (lane == 0) {
                over[atomicAdd(over_ctr, 1ull)] = (uint32_t)R;
                atomicMax(over_ctr + 1, (unsigned long long)nw);
            }
            return;
        }
        rank_row(src, dst, jb, d, comp, base, nw, bm, pre);
    };
    if (BIG) {
        const int64_t rows = (int64_t)over_ctr[0];
        for (int64_t i = warp_id_global(); i < rows; i += warp_count_global()) {
            const int64_t R = (int64_t)over[i], jb = inc_ptr[R];
            long_row(R, jb, inc_ptr[R + 1] - jb);
        }
        return;
    }
    const int64_t groups = (N + per - 1) / per;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t mine = lane < per ? per * g + lane : N;
        int64_t jb = 0, d = 0;
        if (mine < N) {
            jb = inc_ptr[mine];
            d = inc_ptr[mine + 1] - jb;
        }
        if (d == 1) dst[jb] = src[jb];
        // up to eight entries: four rows at a time, eight lanes each
        for (unsigned todo = __ballot_sync(kFull, d >= 2 && d <= 8); todo;) {
            int r = -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int f = todo ? __ffs(todo) - 1 : -1;
                if (lane / 8 == q) r = f;
                todo &= todo - 1;  // 0 stays 0
            }
            const int64_t rj = __shfl_sync(kFull, jb, max(r, 0)), any_d = __shfl_sync(kFull, d, max(r, 0));
            const int rd = r >= 0 ? (int)any_d : 0;
            const bool ok = (lane & 7) < rd;
            const uint2 e = ok ? src[rj + (lane & 7)] : make_uint2(0xffffffffu, 0u);
            int rank = 0;
#pragma unroll
            for (int o = 0; o < 8; ++o) rank += __shfl_sync(kFull, e.x, o, 8) < e.x;
            if (ok) dst[rj + rank] = e;
        }
        for (unsigned todo = __ballot_sync(kFull, d > 8 && d <= kPoolRow); todo; todo &= todo - 1) {
            const int r = __ffs(todo) - 1;
            const int64_t rj = __shfl_sync(kFull, jb, r), rd = __shfl_sync(kFull, d, r);
            if (rd > 32) {
                long_row(per * g + r, rj, rd);
                continue;
            }
            const uint2 e = lane < rd ? src[rj + lane] : make_uint2(0xffffffffu, 0u);
            int rank = 0;
            for (int o = 0; o < (int)rd; ++o) rank += __shfl_sync(kFull, e.x, o) < e.x;
            if (lane < rd) dst[rj + rank] = e;
        }
    }
    spread_rows(
        N, [&](int64_t R) { return inc_ptr[R + 1] - inc_ptr[R] > kPoolRow; },
        [&](int64_t R) { long_row(R, inc_ptr[R], inc_ptr[R + 1] - inc_ptr[R]); });
}

// ---- (3,4): the triangles of every edge, and the 4-cliques of every triangle --
// The list of edge (u,v) holds every triangle on it, by third vertex: the
// common neighbours of u and v, one warp per edge.  Third vertices above v
// make the canonical triangles (u < v < w, lexicographic, grouped by edge in
// tri_ptr / tri_w / tri_e).  A triangle stands in the lists of its three edges.
// The 4-cliques of triangle {u,v,w} are then the z in all three of them: one
// warp per triangle intersects the lists, which are far shorter than the
// neighbourhoods (a planted clique of k vertices: k - 2), and writes its row in
// order of z, with no atomics, no cursors and no search for triangle ids.
// Listing every 4-clique once by degree orientation, with three id searches
// each and a scatter into four rows, took 18.5 ms for 55M 4-cliques (Chung-Lu
// 100K with planted cliques) and left the rows unordered.
template <bool FILL>
__global__ void __launch_bounds__(kThreads) k_edge_lists(int64_t m, const int64_t* __restrict__ rp,
                                                         const int32_t* __restrict__ col,
                                                         const uint32_t* __restrict__ eid,
                                                         const int32_t* __restrict__ e_u,
                                                         const int32_t* __restrict__ e_v, int64_t* __restrict__ lptr,
                                                         int64_t* __restrict__ tri_ptr, int32_t* __restrict__ lw,
                                                         uint32_t* __restrict__ lid, int32_t* __restrict__ tri_w,
                                                         uint32_t* __restrict__ tri_e, uint32_t* __restrict__ te,
                                                         uint32_t* __restrict__ t_pos) {
    __shared__ int32_t bufs[kThreads / 32][nd_list_cursor::kBlock];
    const int lane = threadIdx.x & 31;
    for (int64_t e = warp_id_global(); e < m; e += warp_count_global()) {
        const int32_t u = e_u[e], v = e_v[e];
        const int64_t ub = rp[u], ue = rp[u + 1], vb = rp[v], ve = rp[v + 1];
        const bool us = ue - ub <= ve - vb;  // walk the shorter list
        const int64_t sb = us ? ub : vb, lb = us ? vb : ub;
        const int sn = (int)(us ? ue - ub : ve - vb), ln = (int)(us ? ve - vb : ue - ub);
        const int64_t out = FILL ? lptr[e] : 0, tri = FILL ? tri_ptr[e] : 0;
        int64_t cnt = 0, up = 0;
        nd_list_cursor cur;
        cur.start(col + lb, ln, sn, bufs[threadIdx.x >> 5]);
        for (int j0 = 0; j0 < sn; j0 += 32) {
            const int j = j0 + lane;
            const int32_t w = j < sn ? __ldg(col + sb + j) : 0;
            const int k = cur.find(w, j < sn, __reduce_max_sync(kFull, w));
            const unsigned all = __ballot_sync(kFull, k >= 0), high = __ballot_sync(kFull, k >= 0 && w > v);
            if (FILL && k >= 0) {
                const int64_t slot = out + cnt + __popc(all & lanemask_lt());
                lw[slot] = w;
                if (w > v) {
                    const int64_t id = tri + up + __popc(high & lanemask_lt());
                    lid[slot] = (uint32_t)id;
                    tri_w[id] = w;
                    tri_e[id] = (uint32_t)e;
                    te[3 * id] = (uint32_t)e;
                    if (t_pos) t_pos[3 * id] = (uint32_t)slot;
                } else {
                    // the edge {u,w}, whose list of canonical triangles holds
                    // this one (k_list_ids)
                    lid[slot] = __ldg(eid + (us ? sb + j : lb + k));
                }
            }
            cnt += __popc(all);
            up += __popc(high);
        }
        if (!FILL && lane == 0) {
            lptr[e] = cnt;
            tri_ptr[e] = up;
        }
        __syncwarp();
    }
}

// the ids of the list entries whose third vertex w is below v: v's place among
// the canonical triangles of the edge {u,w} (left in lid)
__global__ void k_list_ids(int64_t m, const int32_t* __restrict__ e_u, const int32_t* __restrict__ e_v,
                           const int64_t* __restrict__ lptr, const int32_t* __restrict__ lw,
                           uint32_t* __restrict__ lid, const int64_t* __restrict__ tri_ptr,
                           const int32_t* __restrict__ tri_w, uint32_t* __restrict__ te,
                           uint32_t* __restrict__ t_pos) {
    const int lane = threadIdx.x & 31;
    for (int64_t e = warp_id_global(); e < m; e += warp_count_global()) {
        const int64_t b = lptr[e], low = (lptr[e + 1] - b) - (tri_ptr[e + 1] - tri_ptr[e]);
        if (low == 0) continue;
        const int32_t u = e_u[e], v = e_v[e];
        for (int64_t s = b + lane; s < b + low; s += 32) {
            const int32_t w = lw[s];
            const uint32_t o = lid[s];
            const int64_t id = lower_bound_i32(tri_w, tri_ptr[o], tri_ptr[o + 1], v);
            lid[s] = (uint32_t)id;
            const int64_t at = 3 * id + (w < u ? 2 : 1);
            te[at] = (uint32_t)e;
            if (t_pos) t_pos[at] = (uint32_t)s;
        }
    }
}

// The 4-cliques of every triangle.  FILL: its row, three runs of d words (the
// slot of z in each of the three lists, or the triangle there: IDS), ordered
// by z; else their number.  Eight triangles per warp at a time: their list
// bounds, a chain of two loads, are fetched by eight lanes at once.
template <bool FILL, bool IDS>
__global__ void __launch_bounds__(kThreads) k_k4_rows(int64_t T, const uint32_t* __restrict__ te,
                                                      const int64_t* __restrict__ lptr,
                                                      const int32_t* __restrict__ lw,
                                                      const uint32_t* __restrict__ lid,
                                                      int64_t* __restrict__ inc_ptr, uint32_t* __restrict__ inc) {
    __shared__ int32_t bufs[kThreads / 32][2][nd_list_cursor::kBlock];
    const int lane = threadIdx.x & 31;
    constexpr int kAtOnce = 8;
    const int64_t groups = (T + kAtOnce - 1) / kAtOnce;
    for (int64_t g = warp_id_global(); g < groups; g += warp_count_global()) {
        const int64_t t0 = g * kAtOnce;
        int64_t b[3] = {0, 0, 0}, jb = 0;  // shortest list first
        int n[3] = {0, 0, 0}, d = 0;
        bool run = lane < kAtOnce && t0 + lane < T;
        if (run && FILL) {
            jb = inc_ptr[t0 + lane];
            d = (int)(inc_ptr[t0 + lane + 1] - jb);
            run = d > 0;
        }
        if (run) {
            uint32_t e[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) e[i] = __ldg(te + 3 * (t0 + lane) + i);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                b[i] = __ldg(lptr + e[i]);
                n[i] = (int)(__ldg(lptr + e[i] + 1) - b[i]);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {  // sort by length: (0,1), (1,2), (0,1)
                const int x = i & 1, y = x + 1;
                if (n[x] > n[y]) {
                    const int tn = n[x];
                    n[x] = n[y];
                    n[y] = tn;
                    const int64_t tb = b[x];
                    b[x] = b[y];
                    b[y] = tb;
                }
            }
        }
        int count = 0;  // lane l: 4-cliques of triangle t0 + l
        // every list holds the triangle's own third vertex, so a 4-clique needs two
        for (unsigned todo = __ballot_sync(kFull, run && n[0] > 1); todo; todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            int64_t lb[3];
            int ln[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                lb[i] = __shfl_sync(kFull, b[i], l);
                ln[i] = __shfl_sync(kFull, n[i], l);
            }
            uint32_t* row = nullptr;
            int rd = 0;
            if (FILL) {
                row = inc + 3 * __shfl_sync(kFull, jb, l);
                rd = __shfl_sync(kFull, d, l);
            }
            nd_list_cursor B, C;
            B.start(lw + lb[1], ln[1], ln[0], bufs[threadIdx.x >> 5][0]);
            C.start(lw + lb[2], ln[2], ln[0], bufs[threadIdx.x >> 5][1]);
            int cnt = 0;
            for (int j0 = 0; j0 < ln[0]; j0 += 32) {
                const int j = j0 + lane;
                const int32_t z = j < ln[0] ? __ldg(lw + lb[0] + j) : 0;
                const int32_t top = __reduce_max_sync(kFull, z);
                const int kb = B.find(z, j < ln[0], top);
                if (!__any_sync(kFull, kb >= 0)) continue;
                const int kc = C.find(z, kb >= 0, top);
                const unsigned hit = __ballot_sync(kFull, kc >= 0);
                if (FILL && kc >= 0) {
                    const int at = cnt + __popc(hit & lanemask_lt());
                    const int64_t s0 = lb[0] + j, s1 = lb[1] + kb, s2 = lb[2] + kc;
                    row[at] = IDS ? lid[s0] : (uint32_t)s0;
                    row[at + rd] = IDS ? lid[s1] : (uint32_t)s1;
                    row[at + 2 * (int64_t)rd] = IDS ? lid[s2] : (uint32_t)s2;
                }
                cnt += __popc(hit);
            }
            if (lane == l) count = cnt;
            __syncwarp();
        }
        if (!FILL && lane < kAtOnce && t0 + lane < T) inc_ptr[t0 + lane] = count;
    }
}

// ---- degree buckets --------------------------------------------------------
// bucket of a row of length d under thresholds t = (t0, t1, t2):
// [1,t0] -> 4 lanes, (t0,t1] -> 8 lanes, (t1,t2] -> a warp, > t2 -> a CTA
__device__ __forceinline__ int bucket_of(int64_t d, int3 t) {
    return d == 0 ? -1 : (d <= t.x ? 0 : (d <= t.y ? 1 : (d <= t.z ? 2 : 3)));
}

// rows per block: kThreads at a time, in order
constexpr int kBucketTile = 2048;

// cnt[b * nblocks + block] = rows of the block's tile in bucket b
__global__ void __launch_bounds__(kThreads) k_bucket_count(int64_t N, const int64_t* __restrict__ inc_ptr, int3 thr,
                                                           int64_t nblocks, int64_t* __restrict__ cnt) {
    __shared__ unsigned c[ND_NB];
    if (threadIdx.x < ND_NB) c[threadIdx.x] = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * kBucketTile;
    unsigned own[ND_NB] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < kBucketTile / kThreads; ++k) {
        const int64_t i = t0 + k * kThreads + threadIdx.x;
        const int b = i < N ? bucket_of(inc_ptr[i + 1] - inc_ptr[i], thr) : -1;
#pragma unroll
        for (int q = 0; q < ND_NB; ++q) own[q] += (b == q);
    }
#pragma unroll
    for (int q = 0; q < ND_NB; ++q) {
        const unsigned w = __reduce_add_sync(kFull, own[q]);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(&c[q], w);
    }
    __syncthreads();
    if (threadIdx.x < ND_NB) cnt[threadIdx.x * nblocks + blockIdx.x] = c[threadIdx.x];
}

// the work items of the tile's rows, in order inside their bucket: start of
// (bucket, block) in off, plus the earlier rows of the bucket in the tile
__global__ void __launch_bounds__(kThreads) k_bucket_scatter(int64_t N, const int64_t* __restrict__ inc_ptr, int3 thr,
                                                             int64_t nblocks, const int64_t* __restrict__ off,
                                                             nd_item* __restrict__ items) {
    constexpr int kWarps = kThreads / 32;
    __shared__ unsigned wcnt[2][kWarps][ND_NB];  // two rounds' buffers: one barrier per round
    int64_t run[ND_NB];
#pragma unroll
    for (int q = 0; q < ND_NB; ++q) run[q] = off[q * nblocks + blockIdx.x];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * kBucketTile;
    for (int k = 0; k < kBucketTile / kThreads && t0 + k * kThreads < N; ++k) {
        const int64_t i = t0 + k * kThreads + threadIdx.x;
        int64_t jb = 0, d = 0;
        if (i < N) {
            jb = inc_ptr[i];
            d = inc_ptr[i + 1] - jb;
        }
        const int b = i < N ? bucket_of(d, thr) : -1;
        unsigned before = 0;
#pragma unroll
        for (int q = 0; q < ND_NB; ++q) {
            const unsigned m = __ballot_sync(kFull, b == q);
            if (b == q) before = __popc(m & lanemask_lt());
            if (lane == 0) wcnt[k & 1][w][q] = __popc(m);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < ND_NB; ++q) {
            unsigned mine = 0, all = 0;
#pragma unroll
            for (int v = 0; v < kWarps; ++v) {
                const unsigned c = wcnt[k & 1][v][q];
                all += c;
                if (v < w) mine += c;
            }
            if (b == q) {
                nd_item it;
                it.jb = jb;
                it.R = (uint32_t)i;
                it.d = (uint32_t)d;
                items[run[q] + mine + before] = it;
            }
            run[q] += all;
        }
    }
}

// graph index of r-clique R (caller's order): the i with off[i] <= R < off[i+1]
__global__ void k_graph_ids(int64_t N, const int64_t* __restrict__ off, int count, const int32_t* __restrict__ to_new,
                            uint32_t* __restrict__ gid) {
    for (int64_t R = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; R < N; R += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = count;  // last i with off[i] <= R
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= R) lo = mid; else hi = mid;
        }
        gid[to_new ? to_new[R] : R] = (uint32_t)lo;
    }
}

__global__ void k_r_cliques(int r, int64_t N, const int32_t* __restrict__ e_u,
                            const int32_t* __restrict__ e_v, const int32_t* __restrict__ tri_w,
                            const uint32_t* __restrict__ tri_e, int32_t* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (r == 1) {
            out[i] = (int32_t)i;
        } else if (r == 2) {
            out[2 * i] = e_u[i];
            out[2 * i + 1] = e_v[i];
        } else {
            uint32_t e = tri_e[i];
            out[3 * i] = e_u[e];
            out[3 * i + 1] = e_v[e];
            out[3 * i + 2] = tri_w[i];
        }
    }
}

// ---- batches: the disjoint union of many graphs (one block per graph) ------
// Vertex ids of graph i are shifted by n_off; its CSR slots by nnz_off.  A
// graph whose offsets or ids fall outside its own range is reported.
__global__ void k_union(const nd_union_part* __restrict__ parts, int count, int64_t* __restrict__ urp,
                        int32_t* __restrict__ ucol, int* __restrict__ err) {
    for (int gi = blockIdx.x; gi < count; gi += gridDim.x) {
        const nd_union_part p = parts[gi];
        if (threadIdx.x == 0 && (p.rp[0] != 0 || p.rp[p.n] != p.nnz)) atomicOr(err, 1);
        for (int64_t i = threadIdx.x; i < p.n; i += blockDim.x) {
            int64_t x = p.rp[i];
            if (x < 0 || x > p.nnz) { atomicOr(err, 1); x = 0; }
            urp[p.n_off + i] = p.nnz_off + x;
        }
        for (int64_t j = threadIdx.x; j < p.nnz; j += blockDim.x) {
            int32_t v = p.col[j];
            if (v < 0 || v >= p.n) { atomicOr(err, 2); v = 0; }
            ucol[p.nnz_off + j] = v + (int32_t)p.n_off;
        }
    }
}

// out[i] = src[idx[i]] for the r-clique offsets of a batch
__global__ void k_gather_i64(const int64_t* __restrict__ src, const int64_t* __restrict__ idx, int count,
                             int64_t* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        out[i] = src[idx[i]];
}

int grid_cap(const nd_incidence* h) { return (h->sm_count > 0 ? h->sm_count : 152) * 8; }

// device words to the handle's pinned words [at, at + count): valid after the
// next nd_wait, so one wait serves several of them
nd_status fetch(nd_incidence* h, int at, const void* d, int count, cudaStream_t st) {
    ND_CUDA(cudaMemcpyAsync(h->h_read + at, d, sizeof(int64_t) * count, cudaMemcpyDeviceToHost, st));
    return ND_OK;
}

nd_status read_flag(nd_incidence* h, const int* dflag, int* hval, cudaStream_t st) {
    ND_CUDA(cudaMemcpyAsync(h->h_read, dflag, sizeof(int), cudaMemcpyDeviceToHost, st));
    ND_TRY(nd_wait(st));
    *hval = *(const int*)h->h_read;
    return ND_OK;
}

nd_status read_i64(nd_incidence* h, const int64_t* d, int64_t* hv, cudaStream_t st) {
    ND_TRY(fetch(h, 0, d, 1, st));
    ND_TRY(nd_wait(st));
    *hv = h->h_read[0];
    return ND_OK;
}

}  // namespace

// Copy the caller's CSR into owned device buffers, validate it, split each
// row at its own vertex and derive the canonical edge numbering offsets.
// the rows longer than kLongRow and the offsets of their kLongSeg segments
// (a host scan over the few such rows); kept on the handle for the edge ids
static nd_status find_long_rows(nd_incidence* h, cudaStream_t st) {
    h->long_count = h->long_segs = 0;
    // a simple graph of n vertices has no row past n - 1 entries; the
    // validation refuses one that is longer
    if (h->n <= kLongRow || h->nnz <= kLongRow) return ND_OK;
    const int64_t cap = h->nnz / kLongRow + 1;
    ND_TRY(nd_alloc((void**)&h->long_rows, sizeof(int32_t) * cap, st, h));
    nd_tmp<int64_t> len(st);
    nd_tmp<unsigned long long> cnt(st);
    ND_TRY(len.alloc(cap));
    ND_TRY(cnt.alloc(1));
    ND_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st));
    k_long_rows<<<nd_blocks_for(h->n, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(
        h->n, h->nnz, h->rp, h->long_rows, len, (unsigned long long)cap, cnt);
    ND_CUDA(cudaGetLastError());
    int64_t cc = 0;
    ND_TRY(read_i64(h, (const int64_t*)cnt.p, &cc, st));
    const unsigned long long c = (unsigned long long)cc;
    if (c > (unsigned long long)cap) {  // overlapping rows: not an offset array
        nd_set_error("row_ptr is not a valid offset array");
        return ND_E_INVAL;
    }
    if (c == 0) return ND_OK;
    std::vector<int64_t> hl(c), off(c + 1, 0);
    ND_CUDA(cudaMemcpyAsync(hl.data(), len.p, sizeof(int64_t) * c, cudaMemcpyDeviceToHost, st));
    ND_TRY(nd_wait(st));
    for (unsigned long long i = 0; i < c; ++i) off[i + 1] = off[i] + (hl[i] + kLongSeg - 1) / kLongSeg;
    ND_TRY(nd_alloc((void**)&h->long_seg, sizeof(int64_t) * (c + 1), st, h));
    ND_CUDA(cudaMemcpyAsync(h->long_seg, off.data(), sizeof(int64_t) * (c + 1), cudaMemcpyHostToDevice, st));
    ND_TRY(nd_wait(st));  // off is a host temporary
    h->long_count = (int64_t)c;
    h->long_segs = off[c];
    return ND_OK;
}

static void release_long_rows(nd_incidence* h, cudaStream_t st) {
    nd_release(h->long_rows, st);
    nd_release(h->long_seg, st);
    h->long_rows = nullptr;
    h->long_seg = nullptr;
    h->long_count = h->long_segs = 0;
}

// validation and degree split of the handle's CSR (h->rp, h->col): nlow,
// up_start, the long rows, for r >= 2 the reverse entries, and h->m
// by_length: the symmetry key of k_validate_split (false only for ids that
// the build assigned by degree class); mirror: record the reverse entries
static nd_status validate_split(nd_incidence* h, cudaStream_t st, bool by_length, bool mirror) {
    const nd_csr gg{h->n, h->nnz, h->rp, h->col, 1};
    const nd_csr* g = &gg;
    ND_TRY(nd_alloc((void**)&h->nlow, sizeof(int32_t) * (g->n > 0 ? g->n : 1), st, h));
    ND_TRY(nd_alloc((void**)&h->up_start, sizeof(int64_t) * (g->n + 1), st, h));
    // reverse entries for the edge ids and the (2,3) adjacency layout (build only)
    if (mirror && h->r >= 2 && g->nnz > 0 && g->nnz < (int64_t)UINT32_MAX)
        ND_TRY(nd_alloc((void**)&h->mirror, sizeof(uint32_t) * g->nnz, st, h));
    // k-core builds (no reverse entries needed) decide symmetry by fingerprint
    const bool fp = h->r == 1;
    nd_tmp<unsigned long long> dsearched(st);
    ND_TRY(dsearched.alloc(4));  // [0] searching entries found, [1..2] fingerprint sums, [3] error bits
    ND_CUDA(cudaMemsetAsync(dsearched, 0, 4 * sizeof(unsigned long long), st));
    int* const derr = (int*)(dsearched.p + 3);
    ND_CUDA(cudaMemsetAsync(h->up_start, 0, sizeof(int64_t) * (g->n + 1), st));
    ND_CUDA(cudaMemsetAsync(h->nlow, 0, sizeof(int32_t) * (g->n > 0 ? g->n : 1), st));
    ND_TRY(find_long_rows(h, st));
    if (g->n > 0) {
        nd_prof_scope ps("validate_split", st);
        const int per = rows_per_warp(h, g->n), blocks = pool_blocks(g->n, per, grid_cap(h) * 4);
        auto split = fp ? k_validate_split<true, true> : (by_length ? k_validate_split<true> : k_validate_split<false>);
        split<<<blocks, kThreads, 0, st>>>(per, g->n, g->nnz, h->rp, h->col, h->nlow, h->up_start, derr, dsearched,
                                           h->mirror, dsearched.p + 1);
        ND_CUDA(cudaGetLastError());
        if (h->long_segs > 0) {
            auto lng = fp ? k_validate_long<true, true> : (by_length ? k_validate_long<true> : k_validate_long<false>);
            lng<<<nd_blocks_for(h->long_segs * 32, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(
                g->n, g->nnz, h->rp, h->col, h->long_rows, h->long_seg, h->long_count, h->long_segs, h->nlow,
                h->up_start, derr, dsearched, h->mirror, dsearched.p + 1);
            ND_CUDA(cudaGetLastError());
        }
    }
    ND_TRY(nd_scan_i64(h->up_start, g->n, st));
    // everything the host decides on, with one wait
    ND_TRY(fetch(h, 0, dsearched.p, 4, st));
    ND_TRY(fetch(h, 4, h->up_start + g->n, 1, st));
    ND_TRY(nd_wait(st));
    const int herr = *(const int*)(h->h_read + 3);
    if (herr) {
        nd_set_error(herr & 1 ? "row_ptr is not a valid offset array"
                              : "col is not simple, sorted and symmetric");
        return ND_E_INVAL;
    }
    const int64_t m = h->h_read[4], found = h->h_read[0];
    const unsigned long long hs[3] = {0, (unsigned long long)h->h_read[1], (unsigned long long)h->h_read[2]};
    if (fp ? (hs[1] != 0 || hs[2] != 0 || 2 * m != g->nnz) : (2 * found != g->nnz || 2 * m != g->nnz)) {
        // every searching entry has its reverse; a surplus of the others is
        // an entry without one
        nd_set_error("col is not symmetric (an entry without its reverse)");
        return ND_E_INVAL;
    }
    h->m = m;
    return ND_OK;
}

// graphs smaller than this keep their ids: their tau fits in cache anyway,
// and the few launches of a relabelling would dominate their build
constexpr int64_t kRelabelMinVertices = 1 << 16;
// words of h_read that the (1,2) relabelling uses past the usual first ones:
// the first id of every class, and the octave bounds on their way up
constexpr int kReadClasses = 8, kReadOctaves = kReadClasses + kClasses - 1;
static_assert(kReadOctaves + 16 <= ND_READ, "the handle's pinned words");

nd_status nd_build_graph(nd_incidence* h, const nd_csr* g, cudaStream_t st, bool truss_relabel) {
    h->n = g->n;
    h->nnz = g->nnz;
    ND_TRY(nd_alloc((void**)&h->rp, sizeof(int64_t) * (g->n + 1), st, h));
    ND_TRY(nd_alloc((void**)&h->col, sizeof(int32_t) * (g->nnz > 0 ? g->nnz : 1), st, h));
    cudaMemcpyKind kind = g->on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    ND_CUDA(cudaMemcpyAsync(h->rp, g->row_ptr, sizeof(int64_t) * (g->n + 1), kind, st));
    if (g->nnz > 0) ND_CUDA(cudaMemcpyAsync(h->col, g->col, sizeof(int32_t) * g->nnz, kind, st));
    // a (2,3) graph that the relabelling will rewrite is validated again
    // under its new ids, and only that second pass records reverse entries
    const bool rewritten = truss_relabel && h->r == 2 && g->n >= kRelabelMinVertices;
    return validate_split(h, st, true, !rewritten);
}

// vertex ids by degree class (k_class_count / k_class_scatter) for the graph
// in h->rp: to_new[caller id] = new id, to_old[new id] = caller id
// read_at >= 0: also fetches the first id of every class to h_read[read_at..]
static nd_status class_ids(nd_incidence* h, int32_t* to_new, int32_t* to_old, cudaStream_t st, int read_at = -1) {
    const int64_t n = h->n;
    const int64_t nblocks = (n + kRelabelTile - 1) / kRelabelTile;
    const int64_t cells = (int64_t)(kClasses - 1) * nblocks;
    nd_tmp<int64_t> cnt(st);
    ND_TRY(cnt.alloc(cells + 1));
    ND_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * (cells + 1), st));
    k_class_count<<<nblocks, kThreads, 0, st>>>(n, h->rp, cnt, nblocks);
    ND_CUDA(cudaGetLastError());
    ND_TRY(nd_scan_i64(cnt, cells, st));
    k_class_scatter<<<nblocks, kThreads, 0, st>>>(n, h->rp, cnt, nblocks, to_new, to_old);
    ND_CUDA(cudaGetLastError());
    if (read_at >= 0)
        ND_CUDA(cudaMemcpy2DAsync(h->h_read + read_at, sizeof(int64_t), cnt.p, sizeof(int64_t) * nblocks,
                                  sizeof(int64_t), kClasses - 1, cudaMemcpyDeviceToHost, st));
    return ND_OK;
}

// (2,3), step 1 of the relabelling (after validation, before the edge ids):
// vertices renumbered by degree class, the graph rewritten under the new ids
// with every row sorted again (a radix sort of the keys (new u, new v) of
// all entries, which is the new CSR in row order), then validated and split
// again.  The caller's CSR and its split are kept until step 2 has mapped
// the edges.  Graphs below kRelabelMinVertices keep their ids.
nd_status nd_relabel_truss_graph(nd_incidence* h, cudaStream_t st) {
    const int64_t n = h->n, nnz = h->nnz;
    if (n < kRelabelMinVertices || h->r != 2) return ND_OK;
    nd_prof_scope ps("relabel", st);
    nd_tmp<int32_t> vto_new(st), ncol(st);
    nd_tmp<int64_t> nrp(st);
    ND_TRY(nd_alloc((void**)&vto_new.p, sizeof(int32_t) * n, st, h));
    ND_TRY(nd_alloc((void**)&h->vto_old, sizeof(int32_t) * n, st, h));
    ND_TRY(class_ids(h, vto_new, h->vto_old, st));
    ND_TRY(nd_alloc((void**)&nrp.p, sizeof(int64_t) * (n + 1), st, h));
    ND_TRY(nd_alloc((void**)&ncol.p, sizeof(int32_t) * (nnz > 0 ? nnz : 1), st, h));
    if (nnz > 0) {
        nd_tmp<unsigned long long> keys(st), alt(st);
        ND_TRY(keys.alloc(nnz));
        ND_TRY(alt.alloc(nnz));
        const int bits = nd_id_bits(n);
        k_relabel_keys<<<nd_blocks_for(n * 32, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(n, h->rp, h->col, vto_new,
                                                                                             bits, keys);
        ND_CUDA(cudaGetLastError());
        if (h->long_segs > 0) {
            k_relabel_keys_long<<<nd_blocks_for(h->long_segs * 32, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(
                h->rp, h->col, vto_new, bits, keys, h->long_rows, h->long_seg, h->long_count, h->long_segs);
            ND_CUDA(cudaGetLastError());
        }
        unsigned long long* sorted = nullptr;
        ND_TRY(nd_sort_u64(keys, alt, nnz, 2 * bits, &sorted, st));
        k_keys_to_col<<<nd_blocks_for(nnz, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(nnz, sorted, bits, ncol);
        ND_CUDA(cudaGetLastError());
    }
    ND_CUDA(cudaMemsetAsync(nrp + n, 0, sizeof(int64_t), st));
    k_new_degrees<<<nd_blocks_for(n, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(n, h->rp, vto_new, nrp);
    ND_CUDA(cudaGetLastError());
    ND_TRY(nd_scan_i64(nrp, n, st));
    nd_release(vto_new.take(), st);
    // keep the caller's graph and split for the edge map; the new graph
    // takes their place and is split again
    h->c_rp = h->rp;
    h->c_col = h->col;
    h->c_nlow = h->nlow;
    h->c_up = h->up_start;
    h->rp = nrp.take();
    h->col = ncol.take();
    h->nlow = nullptr;
    h->up_start = nullptr;
    nd_release(h->mirror, st);
    h->mirror = nullptr;
    release_long_rows(h, st);
    const int64_t m = h->m;
    ND_TRY(validate_split(h, st, false, true));
    if (h->m != m) { nd_set_error("relabelled graph lost edges (internal fault)"); return ND_E_CUDA; }
    return ND_OK;
}

// (2,3), step 2 (after the edge ids of the new graph): the map between the
// new canonical edge ids and the caller's, by searching each new edge's
// caller endpoints in the caller's rows; then the caller's arrays go
nd_status nd_relabel_truss_edges(nd_incidence* h, cudaStream_t st) {
    if (!h->c_rp) return ND_OK;
    const int64_t m = h->m;
    ND_TRY(nd_alloc((void**)&h->to_new, sizeof(int32_t) * (m > 0 ? m : 1), st, h));
    ND_TRY(nd_alloc((void**)&h->to_old, sizeof(int32_t) * (m > 0 ? m : 1), st, h));
    nd_tmp<int> derr(st);
    ND_TRY(derr.alloc(1));
    ND_CUDA(cudaMemsetAsync(derr, 0, sizeof(int), st));
    if (m > 0) {
        nd_prof_scope ps("relabel", st);
        k_edge_map<<<nd_blocks_for(m, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(
            m, h->e_u, h->e_v, h->vto_old, h->c_rp, h->c_col, h->c_nlow, h->c_up, h->to_new, h->to_old, derr);
        ND_CUDA(cudaGetLastError());
    }
    int herr = 0;
    ND_TRY(read_flag(h, derr, &herr, st));
    if (herr) { nd_set_error("an edge of the relabelled graph is missing from the caller's (internal fault)"); return ND_E_CUDA; }
    nd_release(h->c_rp, st);
    nd_release(h->c_col, st);
    nd_release(h->c_nlow, st);
    nd_release(h->c_up, st);
    h->c_rp = h->c_up = nullptr;
    h->c_col = h->c_nlow = nullptr;
    return ND_OK;
}

// the rows of h->rp too long for one warp, as segments
struct nd_row_segments {
    nd_tmp<int32_t> rows;
    nd_tmp<int64_t> off;
    int64_t listed = 0, segs = 0;
    explicit nd_row_segments(cudaStream_t st) : rows(st), off(st) {}
    // waits once, for what has been fetched before too
    nd_status list(nd_incidence* h, cudaStream_t st) {
        const int64_t cap = h->nnz / kSortRow + 1;
        nd_tmp<unsigned long long> count(st);
        ND_TRY(rows.alloc(cap));
        ND_TRY(off.alloc(cap + 1));
        ND_TRY(count.alloc(1));
        ND_CUDA(cudaMemsetAsync(off, 0, sizeof(int64_t) * (cap + 1), st));
        ND_CUDA(cudaMemsetAsync(count, 0, sizeof(unsigned long long), st));
        k_sort_list<<<nd_blocks_for(h->n, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(h->n, h->rp, rows, off, count);
        ND_CUDA(cudaGetLastError());
        ND_TRY(nd_scan_i64(off, cap, st));
        ND_TRY(fetch(h, 0, count.p, 1, st));
        ND_TRY(fetch(h, 1, off.p + cap, 1, st));
        ND_TRY(nd_wait(st));
        listed = h->h_read[0];
        segs = h->h_read[1];
        return ND_OK;
    }
};

// every row of h->rp in the order of k's buckets
template <typename K>
static nd_status order_rows(nd_incidence* h, const K& k, const nd_row_segments& sg, cudaStream_t st) {
    const int per = rows_per_warp(h, h->n);
    k_order_rows<K><<<pool_blocks(h->n, per, grid_cap(h) * 4), kThreads, 0, st>>>(per, h->n, h->rp, k);
    ND_CUDA(cudaGetLastError());
    if (sg.segs == 0) return ND_OK;
    const int blocks = nd_blocks_for(sg.segs * 32, kThreads, grid_cap(h) * 4);
    nd_tmp<int64_t> cells(st);
    ND_TRY(cells.alloc(32 * sg.segs + 1));
    ND_CUDA(cudaMemsetAsync(cells.p + 32 * sg.segs, 0, sizeof(int64_t), st));
    k_sort_count<K><<<blocks, kThreads, 0, st>>>(h->rp, k, sg.rows, sg.off, sg.listed, sg.segs, cells);
    ND_CUDA(cudaGetLastError());
    ND_TRY(nd_scan_i64(cells, 32 * sg.segs, st));
    k_sort_scatter<K><<<blocks, kThreads, 0, st>>>(h->rp, k, sg.rows, sg.off, sg.listed, sg.segs, cells);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

nd_status nd_rows_by_degree(nd_incidence* h, int32_t* vertex, uint32_t* slot, cudaStream_t st) {
    nd_row_segments segments(st);
    ND_TRY(segments.list(h, st));
    return order_rows(h, DegreeOrder{h->rp, h->col, vertex, slot}, segments, st);
}

nd_status nd_relabel_by_degree(nd_incidence* h, cudaStream_t st) {
    const int64_t n = h->n, nnz = h->nnz;
    if (n >= kRelabelMinVertices) {
        nd_prof_scope ps("relabel", st);
        ND_TRY(nd_alloc((void**)&h->to_new, sizeof(int32_t) * n, st, h));
        ND_TRY(nd_alloc((void**)&h->to_old, sizeof(int32_t) * n, st, h));
        ND_TRY(class_ids(h, h->to_new, h->to_old, st, kReadClasses));
        nd_row_segments segments(st);
        ND_TRY(segments.list(h, st));
        // the largest degree in octave o and past it: that of the class of its first id
        int32_t* const oct_max = (int32_t*)(h->h_read + kReadOctaves);
        for (int o = 0; o < 32; ++o) {
            const int64_t id = o > 0 ? (int64_t)1 << o : 0;  // octave 0 holds ids 0 and 1
            int k = -1;
            while (k + 1 < kClasses - 1 && h->h_read[kReadClasses + k + 1] <= id) ++k;
            oct_max[o] = id >= n || k == 32 ? 0 : (k <= 0 ? INT32_MAX : (int32_t)(((int64_t)1 << (32 - k)) - 1));
        }
        ND_TRY(nd_alloc((void**)&h->oct_max, sizeof(int32_t) * 32, st, h));
        ND_CUDA(cudaMemcpyAsync(h->oct_max, oct_max, sizeof(int32_t) * 32, cudaMemcpyHostToDevice, st));
        nd_tmp<int64_t> nrp(st);
        nd_tmp<int32_t> ncol(st);
        ND_TRY(nd_alloc((void**)&nrp.p, sizeof(int64_t) * (n + 1), st, h));
        ND_CUDA(cudaMemsetAsync(nrp + n, 0, sizeof(int64_t), st));
        k_new_degrees<<<nd_blocks_for(n, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(n, h->rp, h->to_new, nrp);
        ND_CUDA(cudaGetLastError());
        ND_TRY(nd_scan_i64(nrp, n, st));
        ND_TRY(nd_alloc((void**)&ncol.p, sizeof(int32_t) * (nnz > 0 ? nnz : 1), st, h));
        if (nnz > 0) ND_TRY(order_rows(h, NewIdOrder{h->col, h->to_new, nrp, ncol}, segments, st));
        nd_release(h->rp, st);
        nd_release(h->col, st);
        h->rp = nrp.take();
        h->col = ncol.take();
    }
    release_long_rows(h, st);
    return ND_OK;
}

nd_status nd_permute_i32(const int32_t* idx, const int32_t* in, int32_t* out, int64_t n, bool scatter,
                         cudaStream_t st) {
    if (n == 0) return ND_OK;
    k_permute_i32<<<nd_blocks_for(n, kThreads, 152 * 8), kThreads, 0, st>>>(n, idx, in, out, scatter ? 1 : 0);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

nd_status nd_build_edges(nd_incidence* h, cudaStream_t st) {
    if (h->m >= (int64_t)UINT32_MAX) { nd_set_error("more than 2^32-1 edges"); return ND_E_TOO_LARGE; }
    ND_TRY(nd_alloc((void**)&h->eid, sizeof(uint32_t) * (h->nnz > 0 ? h->nnz : 1), st, h));
    ND_TRY(nd_alloc((void**)&h->e_u, sizeof(int32_t) * (h->m > 0 ? h->m : 1), st, h));
    ND_TRY(nd_alloc((void**)&h->e_v, sizeof(int32_t) * (h->m > 0 ? h->m : 1), st, h));
    if (h->r == 2) {
        // (2,3) incidence entries are CSR positions (uint32)
        if (h->nnz >= (int64_t)UINT32_MAX) {
            nd_set_error("(2,3) needs fewer than 2^32-1 CSR entries");
            return ND_E_TOO_LARGE;
        }
        h->adj = true;
        ND_TRY(nd_alloc((void**)&h->e_pos, sizeof(uint2) * (h->m > 0 ? h->m : 1), st, h));
    }
    if (h->n > 0 && h->nnz > 0) {
        nd_prof_scope ps("edge_ids", st);
        int blocks = nd_blocks_for(h->n * 32, kThreads, grid_cap(h) * 4);
        k_edge_ids<<<blocks, kThreads, 0, st>>>(h->n, h->rp, h->col, h->nlow, h->up_start, h->eid,
                                                h->e_u, h->e_v, h->mirror, h->e_pos);
        ND_CUDA(cudaGetLastError());
        if (h->long_segs > 0) {
            k_edge_ids_long<<<nd_blocks_for(h->long_segs * 32, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(
                h->rp, h->col, h->nlow, h->up_start, h->eid, h->e_u, h->e_v, h->mirror, h->e_pos, h->long_rows,
                h->long_seg, h->long_count, h->long_segs);
            ND_CUDA(cudaGetLastError());
        }
    }
    release_long_rows(h, st);
    if (!h->adj && h->mirror) {  // only the (2,3) build needs it further
        nd_release(h->mirror, st);
        h->mirror = nullptr;
    }
    return ND_OK;
}

// oriented out-lists (degree order) of the (2,3) build
struct nd_oriented {
    nd_tmp<int64_t> out_ptr;
    nd_tmp<int32_t> out_col, out_src;
    nd_tmp<uint32_t> out_eid;
    nd_tmp<uint2> out_pm;  // CSR positions of the entry and of its reverse
    explicit nd_oriented(cudaStream_t st)
        : out_ptr(st), out_col(st), out_src(st), out_eid(st), out_pm(st) {}
};

static nd_status orient_graph(nd_incidence* h, nd_oriented* o, cudaStream_t st) {
    const int64_t n = h->n, m = h->m;
    ND_TRY(o->out_ptr.alloc(n + 1));
    ND_TRY(o->out_col.alloc(m));
    ND_TRY(o->out_src.alloc(m));
    ND_TRY(o->out_eid.alloc(m));
    const bool positions = h->adj && !h->otf;  // only the stored (2,3) fill uses them
    if (positions) ND_TRY(o->out_pm.alloc(m));
    ND_CUDA(cudaMemsetAsync(o->out_ptr.p + n, 0, sizeof(int64_t), st));
    const int per = rows_per_warp(h, n), vblocks = pool_blocks(n, per, grid_cap(h) * 4);
    if (n > 0) {
        nd_prof_scope ps("orient", st);
        k_orient<false><<<vblocks, kThreads, 0, st>>>(per, n, h->rp, h->col, h->eid, o->out_ptr, nullptr, nullptr, nullptr,
                                                      nullptr, nullptr);
        ND_CUDA(cudaGetLastError());
    }
    ND_TRY(nd_scan_i64(o->out_ptr, n, st));
    if (n > 0) {
        nd_prof_scope ps("orient", st);
        k_orient<true><<<vblocks, kThreads, 0, st>>>(per, n, h->rp, h->col, h->eid, o->out_ptr, o->out_col, o->out_eid,
                                                     o->out_src, h->mirror, positions ? o->out_pm.p : nullptr);
        ND_CUDA(cudaGetLastError());
    }
    return ND_OK;
}

// order the rows of the (2,3) adjacency layout by w (see k_row_rank); if
// the second buffer does not fit, the rows stay in fill order (the h-index
// does not depend on it; the gathers are only less local)
static nd_status sort_tri_rows(nd_incidence* h, cudaStream_t st) {
    const int64_t N = h->num_r, M = h->num_inc;
    nd_tmp<uint2> dst(st);
    if (dst.alloc(M) != ND_OK) {
        nd_set_error("");
        return ND_OK;
    }
    nd_tmp<uint32_t> over(st);
    nd_tmp<unsigned long long> over_ctr(st);
    // no adjacency list of n <= 32 * kRankWords vertices needs more words
    const bool can_overflow = h->n > 32 * (int64_t)kRankWords;
    ND_TRY(over.alloc(can_overflow ? N : 1));
    ND_TRY(over_ctr.alloc(2));
    if (can_overflow) ND_CUDA(cudaMemsetAsync(over_ctr, 0, sizeof(unsigned long long) * 2, st));
    const size_t smem = sizeof(uint32_t) * 2 * kRankWords * kRankWarps;
    ND_CUDA(cudaFuncSetAttribute(k_row_rank<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    {
        nd_prof_scope ps("row_rank", st);
        const int per = rows_per_warp(h, N);
        const int blocks = nd_blocks_for((N + per - 1) / per * 32, 32 * kRankWarps, grid_cap(h) * 8);
        k_row_rank<false><<<blocks, 32 * kRankWarps, smem, st>>>(per, N, h->inc_ptr, h->e_u, h->e_v, h->rp,
                                                                  (const uint2*)h->inc, dst, over, over_ctr,
                                                                  nullptr, 0);
        ND_CUDA(cudaGetLastError());
    }
    unsigned long long hc[2] = {0, 0};
    if (can_overflow) {
        ND_TRY(fetch(h, 0, over_ctr.p, 2, st));
        ND_TRY(nd_wait(st));
        hc[0] = (unsigned long long)h->h_read[0];
        hc[1] = (unsigned long long)h->h_read[1];
    }
    if (hc[0] > 0) {
        // rows whose shorter adjacency list needs more than kRankWords words
        const int warps = 64;
        nd_tmp<uint32_t> scratch(st);
        ND_TRY(scratch.alloc((int64_t)2 * (int64_t)hc[1] * warps));
        nd_prof_scope ps("row_rank", st);
        k_row_rank<true><<<warps / kRankWarps, 32 * kRankWarps, 0, st>>>(
            1, N, h->inc_ptr, h->e_u, h->e_v, h->rp, (const uint2*)h->inc, dst, over, over_ctr, scratch,
            (int64_t)hc[1]);
        ND_CUDA(cudaGetLastError());
    }
    nd_release(h->inc, st);
    h->inc = reinterpret_cast<uint32_t*>(dst.take());
    h->rows_sorted = true;
    return ND_OK;
}

// smaller (2,3) builds search twice: their searches are a few microseconds,
// less than the launches, the scan and the wait that size the records
constexpr int64_t kRecordMinEdges = 1 << 16;

nd_status nd_build_tri_incidence(nd_incidence* h, cudaStream_t st) {
    const int64_t m = h->m;
    h->num_r = m;
    ND_TRY(nd_alloc((void**)&h->inc_ptr, sizeof(int64_t) * (m + 1), st, h));
    ND_CUDA(cudaMemsetAsync(h->inc_ptr, 0, sizeof(int64_t) * (m + 1), st));
    if (m == 0) { h->num_inc = 0; ND_TRY(nd_alloc((void**)&h->inc, 16, st, h)); return ND_OK; }
    nd_oriented o(st);
    ND_TRY(orient_graph(h, &o, st));
    const int eblocks = nd_blocks_for(m * 32, kThreads, grid_cap(h) * 4);  // a warp per oriented edge
    const int per = rows_per_warp(h, m), pblocks = pool_blocks(m, per, grid_cap(h) * 4);
    // the stored adjacency layout keeps the count pass's triangles as records
    // (4 B each, min(|out(u)|, |out(v)|) slots reserved per oriented edge), so
    // that the fill does not search again; without the memory for them the
    // fill searches as the count pass does
    nd_tmp<int64_t> rec_ptr(st);
    nd_tmp<uint32_t> rec(st), rec_cnt(st);
    bool use_rec = false;
    if (h->adj && !h->otf && m >= kRecordMinEdges && rec_ptr.alloc(m + 1) == ND_OK) {
        k_rec_bound<<<nd_blocks_for(m, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(m, o.out_ptr, o.out_src,
                                                                                     o.out_col, rec_ptr);
        ND_CUDA(cudaGetLastError());
        ND_CUDA(cudaMemsetAsync(rec_ptr.p + m, 0, sizeof(int64_t), st));
        ND_TRY(nd_scan_i64(rec_ptr, m, st));
        int64_t slots = 0;
        ND_TRY(read_i64(h, rec_ptr.p + m, &slots, st));
        use_rec = rec.alloc(slots) == ND_OK && rec_cnt.alloc(m) == ND_OK;
        if (!use_rec) nd_set_error("");
    }
    {
        // per-edge counts fit 32 bits (d_s < n); 32-bit atomics, widened for the scan
        nd_tmp<unsigned> cnt32(st);
        ND_TRY(cnt32.alloc(m));
        ND_CUDA(cudaMemsetAsync(cnt32, 0, sizeof(unsigned) * m, st));
        nd_prof_scope ps("tri_count", st, 2);
        auto count = use_rec ? k_tri_count<true> : k_tri_count<false>;
        count<<<pblocks, kThreads, 0, st>>>(
            per, m, o.out_ptr, o.out_col, o.out_eid, o.out_src, cnt32.p, use_rec ? rec_ptr.p : nullptr,
            use_rec ? rec.p : nullptr, use_rec ? rec_cnt.p : nullptr);
        ND_CUDA(cudaGetLastError());
        k_widen_u32<<<nd_blocks_for(m, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(m, cnt32, h->inc_ptr);
        ND_CUDA(cudaGetLastError());
    }
    ND_TRY(nd_scan_i64(h->inc_ptr, m, st));
    ND_TRY(read_i64(h, h->inc_ptr + m, &h->num_inc, st));
    if (h->otf) {
        // no stored incidence: the counts (d_s, tau_0 and the buckets) are all
        // that is kept; every pass finds the triangles again
        nd_release(h->mirror, st);
        h->mirror = nullptr;
        return nd_alloc((void**)&h->inc, 16, st, h);
    }
    ND_TRY(nd_alloc((void**)&h->inc, sizeof(uint32_t) * 2 * (h->num_inc > 0 ? h->num_inc : 1), st, h));
    if (h->num_inc > 0) {
        nd_tmp<unsigned long long> cursor(st);
        nd_tmp<unsigned> cursor32(st);
        const bool narrow = h->adj && h->num_inc < (int64_t)UINT32_MAX;  // 32-bit slot atomics
        if (narrow) {
            ND_TRY(cursor32.alloc(m));
            k_narrow_u32<<<nd_blocks_for(m, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(m, h->inc_ptr, cursor32);
            ND_CUDA(cudaGetLastError());
        } else {
            ND_TRY(cursor.alloc(m));
            ND_CUDA(cudaMemcpyAsync(cursor, h->inc_ptr, sizeof(int64_t) * m, cudaMemcpyDeviceToDevice, st));
        }
        nd_prof_scope ps("tri_fill", st);
        if (use_rec && narrow)
            k_tri_fill_rec<unsigned><<<pblocks, kThreads, 0, st>>>(per, m, o.out_ptr, o.out_col, o.out_eid, o.out_src,
                                                                   o.out_pm, cursor32.p, (uint2*)h->inc, rec_ptr, rec,
                                                                   rec_cnt);
        else if (use_rec)
            k_tri_fill_rec<unsigned long long><<<pblocks, kThreads, 0, st>>>(
                per, m, o.out_ptr, o.out_col, o.out_eid, o.out_src, o.out_pm, cursor.p, (uint2*)h->inc, rec_ptr,
                rec, rec_cnt);
        else if (narrow)
            k_tri_fill_search<unsigned><<<eblocks, kThreads, 0, st>>>(m, o.out_ptr, o.out_col, o.out_eid, o.out_src,
                                                                      o.out_pm, cursor32.p, (uint2*)h->inc);
        else
            k_tri_fill_search<unsigned long long><<<eblocks, kThreads, 0, st>>>(m, o.out_ptr, o.out_col, o.out_eid,
                                                                                o.out_src, o.out_pm, cursor.p,
                                                                                (uint2*)h->inc);
        ND_CUDA(cudaGetLastError());
    }
    // the records are no longer needed: free them before the row ranking
    // takes its second incidence buffer
    nd_release(rec.p, st);
    rec.p = nullptr;
    if (h->adj) {
        nd_release(h->mirror, st);  // build only
        h->mirror = nullptr;
        if (h->num_inc > 0) ND_TRY(sort_tri_rows(h, st));
    }
    return ND_OK;
}

// may a (3,4) handle of T triangles and M incidences take the list layout?
// What it holds beyond the id layout must not make a handle miss the memory
// limit that would do without.
static bool list_layout_fits(const nd_incidence* h, int64_t T, int64_t M) {
    const int64_t limit = nd_handle_limit();
    if (limit <= 0) return true;
    const int64_t extra = 24 * T + 12 * T + T;          // t_pos, t_id; two 16-bit copies; frontier bits
    const int64_t rest = 12 * M + 16 * T + 8 * T + 4 * T + (1 << 16);  // incidence, items, tau, a batch's graph ids
    return h->bytes + extra + rest <= limit;
}

nd_status nd_build_k4_incidence(nd_incidence* h, cudaStream_t st) {
    const int64_t m = h->m;
    ND_TRY(nd_alloc((void**)&h->tri_ptr, sizeof(int64_t) * (m + 1), st, h));
    ND_CUDA(cudaMemsetAsync(h->tri_ptr, 0, sizeof(int64_t) * (m + 1), st));
    nd_tmp<int64_t> lptr(st);
    ND_TRY(lptr.alloc(m + 1));
    ND_CUDA(cudaMemsetAsync(lptr, 0, sizeof(int64_t) * (m + 1), st));
    const int eblocks = nd_blocks_for(m * 32, kThreads, grid_cap(h) * 4);
    if (m > 0) {
        nd_prof_scope ps("edge_lists", st);
        k_edge_lists<false><<<eblocks, kThreads, 0, st>>>(m, h->rp, h->col, h->eid, h->e_u, h->e_v, lptr, h->tri_ptr,
                                                          nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
        ND_CUDA(cudaGetLastError());
    }
    ND_TRY(nd_scan_i64(lptr, m, st));
    ND_TRY(nd_scan_i64(h->tri_ptr, m, st));
    ND_TRY(read_i64(h, h->tri_ptr + m, &h->num_tri, st));
    const int64_t T = h->num_tri;
    if (T >= (int64_t)UINT32_MAX) { nd_set_error("more than 2^32-1 triangles"); return ND_E_TOO_LARGE; }
    h->num_r = T;
    ND_TRY(nd_alloc((void**)&h->tri_w, sizeof(int32_t) * (T > 0 ? T : 1), st, h));
    ND_TRY(nd_alloc((void**)&h->tri_e, sizeof(uint32_t) * (T > 0 ? T : 1), st, h));
    ND_TRY(nd_alloc((void**)&h->inc_ptr, sizeof(int64_t) * (T + 1), st, h));
    ND_CUDA(cudaMemsetAsync(h->inc_ptr + T, 0, sizeof(int64_t), st));
    if (T == 0) { h->num_inc = 0; ND_TRY(nd_alloc((void**)&h->inc, 16, st, h)); return ND_OK; }
    nd_tmp<int32_t> lw(st);
    nd_tmp<uint32_t> lid(st), te(st), t_pos(st);
    ND_TRY(lw.alloc(3 * T));
    ND_TRY(lid.alloc(3 * T));
    ND_TRY(te.alloc(3 * T));
    // without the slots, whatever the reason, the rows hold triangle ids
    if (3 * T < (int64_t)UINT32_MAX && t_pos.alloc(3 * T) != ND_OK) nd_set_error("");
    {
        nd_prof_scope ps("edge_lists", st, 2);
        k_edge_lists<true><<<eblocks, kThreads, 0, st>>>(m, h->rp, h->col, h->eid, h->e_u, h->e_v, lptr, h->tri_ptr, lw,
                                                         lid, h->tri_w, h->tri_e, te, t_pos);
        ND_CUDA(cudaGetLastError());
        k_list_ids<<<eblocks, kThreads, 0, st>>>(m, h->e_u, h->e_v, lptr, lw, lid, h->tri_ptr, h->tri_w, te, t_pos);
        ND_CUDA(cudaGetLastError());
    }
    const int tblocks = nd_blocks_for(T * 4, kThreads, grid_cap(h) * 4);
    {
        nd_prof_scope ps("k4_count", st);
        k_k4_rows<false, false><<<tblocks, kThreads, 0, st>>>(T, te, lptr, lw, lid, h->inc_ptr, nullptr);
        ND_CUDA(cudaGetLastError());
    }
    ND_TRY(nd_scan_i64(h->inc_ptr, T, st));
    ND_TRY(read_i64(h, h->inc_ptr + T, &h->num_inc, st));
    const size_t inc_bytes = sizeof(uint32_t) * 3 * (h->num_inc > 0 ? h->num_inc : 1);
    bool slots = t_pos.p && list_layout_fits(h, T, h->num_inc);
    if (!slots || nd_alloc((void**)&h->inc, inc_bytes, st, h) != ND_OK) {
        slots = false;
        nd_release(t_pos.take(), st);  // room for the rows
        ND_TRY(nd_alloc((void**)&h->inc, inc_bytes, st, h));
        nd_set_error("");
    }
    if (h->num_inc > 0) {
        nd_prof_scope ps("k4_fill", st);
        auto fill = slots ? k_k4_rows<true, false> : k_k4_rows<true, true>;
        fill<<<tblocks, kThreads, 0, st>>>(T, te, lptr, lw, lid, h->inc_ptr, h->inc);
        ND_CUDA(cudaGetLastError());
    }
    if (slots) {
        h->t_pos = t_pos.take();
        h->t_id = lid.take();
        h->bytes += (int64_t)sizeof(uint32_t) * 6 * T;
    }
    return ND_OK;
}

nd_status nd_build_buckets(nd_incidence* h, cudaStream_t st) {
    const int64_t N = h->num_r;
    nd_drop_graphs(h);  // they hold the old buckets
    for (int b = 0; b <= ND_NB; ++b) h->bucket_lo[b] = 0;
    h->num_zero = N;
    if (!h->items) ND_TRY(nd_alloc((void**)&h->items, sizeof(nd_item) * (N > 0 ? N : 1), st, h));
    if (N == 0) return ND_OK;
    // a stable counting sort of the rows by bucket: the counts per (bucket,
    // tile), one scan, one scatter, and the five bounds read back at once.
    // One flag array, scan and read-back per bucket before: 0.16 of the 1.1 ms
    // of a 10,000-edge k-truss, and 16 B more per row of scratch.
    const int3 thr = make_int3(h->thr[0], h->thr[1], h->thr[2]);
    const int64_t nblocks = (N + kBucketTile - 1) / kBucketTile;
    nd_tmp<int64_t> cnt(st);
    ND_TRY(cnt.alloc(ND_NB * nblocks + 1));
    {
        nd_prof_scope ps("buckets", st);
        k_bucket_count<<<(unsigned)nblocks, kThreads, 0, st>>>(N, h->inc_ptr, thr, nblocks, cnt);
        ND_CUDA(cudaGetLastError());
    }
    ND_CUDA(cudaMemsetAsync(cnt.p + ND_NB * nblocks, 0, sizeof(int64_t), st));
    ND_TRY(nd_scan_i64(cnt, ND_NB * nblocks, st));
    {
        nd_prof_scope ps("buckets", st);
        k_bucket_scatter<<<(unsigned)nblocks, kThreads, 0, st>>>(N, h->inc_ptr, thr, nblocks, cnt, h->items);
        ND_CUDA(cudaGetLastError());
    }
    // the first entry of every bucket's counts, and the total
    ND_CUDA(cudaMemcpy2DAsync(h->h_read, sizeof(int64_t), cnt.p, sizeof(int64_t) * nblocks, sizeof(int64_t),
                              ND_NB + 1, cudaMemcpyDeviceToHost, st));
    ND_TRY(nd_wait(st));
    for (int b = 0; b <= ND_NB; ++b) h->bucket_lo[b] = h->h_read[b];
    h->num_zero = N - h->bucket_lo[ND_NB];
    return ND_OK;
}

nd_status nd_write_r_cliques(const nd_incidence* h, int32_t* out_dev, cudaStream_t st) {
    if (h->num_r == 0) return ND_OK;
    int blocks = nd_blocks_for(h->num_r, kThreads, grid_cap(h) * 2);
    nd_prof_scope ps("r_cliques", st);
    if (h->r == 2 && h->vto_old)
        k_r_cliques_mapped<<<blocks, kThreads, 0, st>>>(h->num_r, h->e_u, h->e_v, h->vto_old, h->to_old, out_dev);
    else
        k_r_cliques<<<blocks, kThreads, 0, st>>>(h->r, h->num_r, h->e_u, h->e_v, h->tri_w, h->tri_e, out_dev);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

nd_status nd_union_device(const nd_union_part* parts_host, int count, int64_t n, int64_t nnz, int64_t* urp,
                          int32_t* ucol, cudaStream_t st) {
    nd_tmp<nd_union_part> dparts(st);
    nd_tmp<int> derr(st);
    ND_TRY(dparts.alloc(count));
    ND_TRY(derr.alloc(1));
    ND_CUDA(cudaMemsetAsync(derr, 0, sizeof(int), st));
    if (count > 0)
        ND_CUDA(cudaMemcpyAsync(dparts, parts_host, sizeof(nd_union_part) * count, cudaMemcpyHostToDevice, st));
    if (count > 0) {
        nd_prof_scope ps("union", st);
        k_union<<<count < 152 * 16 ? count : 152 * 16, kThreads, 0, st>>>(dparts, count, urp, ucol, derr);
        ND_CUDA(cudaGetLastError());
    }
    ND_CUDA(cudaMemcpyAsync(urp + n, &nnz, sizeof(int64_t), cudaMemcpyHostToDevice, st));
    int herr = 0;
    ND_CUDA(cudaMemcpyAsync(&herr, derr.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    ND_TRY(nd_wait(st));
    if (herr) {
        nd_set_error(herr & 1 ? "a graph of the batch has an invalid row_ptr"
                              : "a graph of the batch has a neighbour id outside its own vertex range");
        return ND_E_INVAL;
    }
    return ND_OK;
}

// r-clique offsets of the graphs of a batch: the union's canonical order
// lists graph 0's r-cliques first, then graph 1's, and so on.
nd_status nd_batch_offsets(const nd_incidence* h, const int64_t* vertex_off /* count+1, host */, int count,
                           int64_t* r_off /* count+1, host */, cudaStream_t st) {
    if (h->r == 1) {
        for (int i = 0; i <= count; ++i) r_off[i] = vertex_off[i];
        return ND_OK;
    }
    nd_tmp<int64_t> didx(st), dout(st);
    ND_TRY(didx.alloc(count + 1));
    ND_TRY(dout.alloc(count + 1));
    ND_CUDA(cudaMemcpyAsync(didx, vertex_off, sizeof(int64_t) * (count + 1), cudaMemcpyHostToDevice, st));
    // edges owned by vertices below the graph's first vertex
    k_gather_i64<<<nd_blocks_for(count + 1, kThreads, 64), kThreads, 0, st>>>(h->up_start, didx, count + 1, dout);
    ND_CUDA(cudaGetLastError());
    const int64_t* res = dout;
    if (h->r == 3) {
        // triangles owned by those edges
        k_gather_i64<<<nd_blocks_for(count + 1, kThreads, 64), kThreads, 0, st>>>(h->tri_ptr, dout, count + 1, didx);
        ND_CUDA(cudaGetLastError());
        res = didx;
    }
    ND_CUDA(cudaMemcpyAsync(r_off, res, sizeof(int64_t) * (count + 1), cudaMemcpyDeviceToHost, st));
    ND_TRY(nd_wait(st));
    return ND_OK;
}

nd_status nd_batch_graph_ids(nd_incidence* h, const int64_t* r_off, int count, cudaStream_t st) {
    if (count < 2 || h->num_r == 0) return ND_OK;  // one graph: nothing to skip
    nd_tmp<int64_t> doff(st);
    ND_TRY(doff.alloc(count + 1));
    ND_CUDA(cudaMemcpyAsync(doff, r_off, sizeof(int64_t) * (count + 1), cudaMemcpyHostToDevice, st));
    ND_TRY(nd_alloc((void**)&h->gid, sizeof(uint32_t) * h->num_r, st, h));
    k_graph_ids<<<nd_blocks_for(h->num_r, kThreads, grid_cap(h) * 4), kThreads, 0, st>>>(h->num_r, doff, count,
                                                                                         h->to_new, h->gid);
    ND_CUDA(cudaGetLastError());
    h->ngraphs = count;
    return nd_wait(st);  // the offsets are a host array
}
