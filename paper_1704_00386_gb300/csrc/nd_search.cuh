// The h-index of one incidence row (Def. 3, clipped to tau(R): Section 4.4): by
// a group of 4 or 8 lanes, a warp, or a CTA.  The passes (nd_hindex.cu) give each of
// them a functor rho(j), the value of entry j, which may be a smaller one every
// time that it is asked: AND lowers tau while rows are read.
// Nothing here but arithmetic, warp intrinsics and shared memory of the
// caller's, so that the routines also compile for the host with those
// intrinsics defined there.
#pragma once

#include <stdint.h>

namespace {

constexpr int kThreads = 256;  // of a pass kernel's block

// What a row's order says about the entries that are still to come.  Rows of a
// relabelled (1,2) graph are ordered by floor(log2 id), and ids by degree
// class, so past an entry of octave o no tau exceeds oct_max[o].
struct NoBound {
    static constexpr bool kOn = false;
    __device__ __forceinline__ bool past(int) const { return false; }
    __device__ __forceinline__ int max_from(int) const { return INT32_MAX; }
};
// the first id from which on no vertex has degree >= h (whole warp)
__device__ __forceinline__ uint32_t id_limit(const int32_t* __restrict__ oct_max, int32_t h) {
    const unsigned m = __ballot_sync(0xffffffffu, __ldg(oct_max + (threadIdx.x & 31)) < h);
    return m ? 1u << (__ffs(m) - 1) : 0xffffffffu;
}
struct IdBound {
    static constexpr bool kOn = true;
    const uint32_t* __restrict__ row;
    const int32_t* __restrict__ oct_max;
    uint32_t limit;  // of the row's tau
    // can no entry from j on reach the row's tau?  (j - 1 has just been read)
    __device__ __forceinline__ bool past(int j) const { return __ldg(row + j - 1) >= limit; }
    // the largest tau from entry j on
    __device__ __forceinline__ int max_from(int j) const { return __ldg(oct_max + 31 - __clz(__ldg(row + j) | 1u)); }
};

// f(rho(j)) for the entries j in [i, end), STEP lanes wide: four loads per
// lane in flight, without tests while whole blocks are left; the rest is one
// block with a test per entry (rho = -1 past the end, which no step counts).
template <int STEP, typename F, typename G>
__device__ __forceinline__ void stream_row(const F& rho, int i, int end, G&& f) {
    const int lane = STEP == 32 ? (threadIdx.x & 31) : threadIdx.x;
    for (; end - i >= 4 * STEP; i += 4 * STEP) {
        int32_t r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = rho(i + u * STEP + lane);
#pragma unroll
        for (int u = 0; u < 4; ++u) f((int)((unsigned)i + u * STEP + lane), r[u]);
    }
    if (end - i > 2 * STEP) {
        int32_t r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned j = (unsigned)i + u * STEP + lane;  // may leave 31 bits
            r[u] = j < (unsigned)end ? rho((int)j) : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) f((int)((unsigned)i + u * STEP + lane), r[u]);
    } else if (end > i) {
        int32_t r[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const unsigned j = (unsigned)i + u * STEP + lane;  // may leave 31 bits
            r[u] = j < (unsigned)end ? rho((int)j) : -1;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) f((int)((unsigned)i + u * STEP + lane), r[u]);
    }
}

// H({rho_j}) clipped to t, for one r-clique per group of G lanes (t = 0 for
// a group without a row); the row (at most G*C <= 64 entries, so t <= 64) is
// held in registers as min(rho, t), four 8-bit values per register.  dmax:
// the longest row of the warp's groups.  Every lane of the warp takes part
// in every step.
template <int G, int C, typename F>
__device__ __forceinline__ int32_t group_hindex(const F& rho, int d, int dmax, int32_t t) {
    static_assert(G * C <= 64, "values fit 7 bits, with one spare for the comparison");
    const int lane = threadIdx.x & (G - 1);
    constexpr int W = (C + 3) / 4;
    constexpr unsigned kHigh = 0x80808080u;
    unsigned pk[W];
    int cnt = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        pk[w] = kHigh;
        if (w == 0 || dmax > 4 * w * G) {  // the same for the whole warp
            int32_t r[4];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (4 * w + c < C) {
                    const int j = lane + (4 * w + c) * G;
                    r[c] = j < d ? rho(j) : 0;
                }
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (4 * w + c < C) {
                    cnt += (r[c] >= t);
                    pk[w] |= (unsigned)max(min(r[c], t), 0) << (8 * c);
                }
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (cnt >= t) cnt = t;
    int lo = cnt, hi = max(t, cnt + 1);  // #{rho >= lo} >= lo holds; at hi it fails (or H = t is settled)
    while (__any_sync(0xffffffffu, hi - lo > 1)) {
        const int mid = (lo + hi) >> 1;  // >= 1 where it is used
        const unsigned m4 = (unsigned)mid * 0x01010101u;
        int c2 = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) c2 += __popc((pk[w] - m4) & kHigh);  // bytes >= mid; no borrow crosses a byte
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        if (hi - lo > 1) {
            if (c2 >= mid) lo = mid; else hi = mid;
        }
    }
    return max(min(lo, t), 0);
}

// the smallest shift that maps [0, span) onto fewer than `bins` values
__device__ __forceinline__ int bin_shift(unsigned span, int bins) {
    const int s = (32 - __clz(span - 1)) - (31 - __clz(bins));
    return span > 1 && s > 0 ? s : 0;
}

// The bin of a histogram that holds H, by one full warp.  Bin b counts rho in
// [lo + (b << shift), lo + ((b + 1) << shift)); `above` counts rho past the
// last bin.  #{rho >= lo + (b << shift)} is above plus the suffix sum from b,
// and H lies in the last bin whose sum reaches its lower edge (bin 0 where none
// does: #{rho >= lo} >= lo has been seen).  Blocks of 128 bins from the top, four
// to a lane; returns the bin, with CARRY also the count past it, in `above`.
// PK: 16-bit counters, bin b in half b / HW of word b % HW.
template <bool PK, int HW, bool CARRY>
__device__ __forceinline__ int select_bin(const unsigned* bins, int lo, int shift, int nb, int& above) {
    const int lane = threadIdx.x & 31;
    for (int c = (nb - 1) >> 7;; --c) {
        const int b0 = 128 * c;
        uint4 w = *reinterpret_cast<const uint4*>(bins + (PK ? (b0 & (HW - 1)) : b0) + 4 * lane);
        if (PK) {
            if (b0 >= HW) w = make_uint4(w.x >> 16, w.y >> 16, w.z >> 16, w.w >> 16);
            else w = make_uint4(w.x & 0xffffu, w.y & 0xffffu, w.z & 0xffffu, w.w & 0xffffu);
        }
        const int s3 = (int)w.w, s2 = s3 + (int)w.z, s1 = s2 + (int)w.y, s0 = s1 + (int)w.x;
        int incl = s0;  // suffix over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_down_sync(0xffffffffu, incl, o);
            if (lane + o < 32) incl += v;
        }
        const int after = above + incl - s0;  // rho past this lane's bins
        // lower edges; unsigned, because those of the padding past nb may leave 31 bits
        const unsigned e0 = (unsigned)lo + ((unsigned)(b0 + 4 * lane) << shift), w1 = 1u << shift;
        int best = -1, past = 0;
        if ((unsigned)(after + s0) >= e0) { best = 0; past = after + s1; }
        if ((unsigned)(after + s1) >= e0 + w1) { best = 1; past = after + s2; }
        if ((unsigned)(after + s2) >= e0 + 2 * w1) { best = 2; past = after + s3; }
        if ((unsigned)(after + s3) >= e0 + 3 * w1) { best = 3; past = after; }
        const unsigned hit = __ballot_sync(0xffffffffu, best >= 0);
        if (hit || c == 0) {
            const int src = hit ? 31 - __clz(hit) : 0;
            if (CARRY) above = __shfl_sync(0xffffffffu, past, src);
            return b0 + 4 * src + max(__shfl_sync(0xffffffffu, best, src), 0);
        }
        above += __shfl_sync(0xffffffffu, incl, 0);
    }
}

// H({rho_j}) clipped to t by one warp, streaming the row.
// count first (direct = false): count rho >= t, reading no further than the
// count still needs: t entries at or above t settle H = t.  Rows are in
// order of the third vertex's degree class where the build renumbers, so the
// entries that reach t come early: at convergence a row is read to about
// 0.58 of its length (R-MAT scale 18 k-truss; the floor, t entries, is 0.47).
// A row that fails is streamed again into a histogram over [count, t).
// direct: straight into the histogram over [0, t) (rows that are expected to
// fail: the early passes, and rows that changed in the pass before).
// The histogram has up to 2 * HW bins (PK: 16-bit counters, two to a word, for
// rows of fewer than 65,536 entries; else HW bins of 32 bits), one per value
// while t allows, so H is exact after one sweep there, and after two for
// longer rows.
// AND lowers tau between the sweeps of a row, so a sweep counts all that its
// sums need: the entries past its bins (ge) too.  With the count of an earlier
// sweep in its place, a neighbour X that fell to x in between would count twice,
// and R would keep an h below x that x does not support: X notifies R only if
// x <= tau(R).  With one sweep's counts, what no longer supports h has fallen
// below h, and so notifies R.  The same holds for lo, the bound of an earlier
// sweep.  (tests/test_row_search.py plays the interleaving.)
// F::kCarry: the values are the same at every reading (SND), and the count is
// carried from sweep to sweep.  That is for (1,2) and (3,4): SND of an R-MAT
// k-core of 16.7M vertices 76.6 against 78.5 ms with a fresh count, Chung-Lu 100K
// (3,4) 40.2 against 41.0; the k-truss counts afresh, R-MAT of 1,048,576 vertices
// 108.9 against 118.4 ms (the kernels spill differently).
// bound: a count also stops where the rest of the row cannot reach t.
template <bool PK, int HW, typename F, typename B>
__device__ __forceinline__ int32_t warp_hindex(const F& rho, const B& bound, int d, int32_t t, bool direct,
                                               unsigned* bins) {
    const int lane = threadIdx.x & 31;
    if (t <= 0) return 0;
    int lo = 0, hi = t, above = 0;
    if (!direct) {
        int cnt = 0, have = 0;
        for (int i = 0; i < d;) {
            const int need = max((min(t - have, 1 << 30) + 31) & ~31, 64);
            const int end = d - i > need ? i + need : d;
            stream_row<32>(rho, i, end, [&](int, int32_t r) { cnt += (r >= t); });
            i = end;
            have = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
            if (have >= t) return t;
            if (bound.past(end)) break;
        }
        lo = above = have;  // #{rho >= lo} >= lo holds; at hi it fails
        if (hi - lo <= 1) return lo;
    }
    for (;;) {
        const unsigned span = (unsigned)(hi - lo);
        const int shift = bin_shift(span, PK ? 2 * HW : HW);
        const int nb = (int)((span - 1) >> shift) + 1;
        for (int i = 0; i < min(nb, HW); i += 128)  // whole blocks of 128, as select_bin reads them
            *reinterpret_cast<uint4*>(bins + i + 4 * lane) = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        int ge = 0;
        stream_row<32>(rho, 0, d, [&](int, int32_t r) {
            const unsigned x = (unsigned)(r - lo);
            if (x < span) {
                const unsigned b = x >> shift;
                if (PK) atomicAdd(bins + (b & (HW - 1)), b < (unsigned)HW ? 1u : 0x10000u);
                else atomicAdd(bins + b, 1u);
            } else {
                ge += (r >= hi);
            }
        });
        __syncwarp();
        if (!F::kCarry) {
            above = (int)__reduce_add_sync(0xffffffffu, (unsigned)ge);
            if (above >= hi) return hi;  // a direct row's first sweep: hi is t
        } else if (direct) {
            above = (int)__reduce_add_sync(0xffffffffu, (unsigned)ge);
            if (above >= t) return t;
            direct = false;
        }
        const int b = select_bin<PK, HW, F::kCarry>(bins, lo, shift, nb, above);
        lo += b << shift;
        hi = min(hi, lo + (1 << shift));
        if (hi - lo <= 1) return lo;
        __syncwarp();
    }
}

// entries of a CTA row between two tests of its count, at least
constexpr int kCtaSegment = 2048;

// The same by the whole CTA (the longest rows): 32-bit counters, as many bins
// as the block's histogram has words; warp 0 selects the bin.  A sweep also
// stops where u, the most the rest of the row can reach, is settled: once
// #{rho >= u} >= u, H is at least u, and the rest, which is below hi, counts for
// no larger value.
// That is what keeps the hub rows of a k-core short: on R-MAT scale 20 the
// rows past 2,048 entries hold 22% of all entries, and a search needs a third
// of those, a converged count an eighth.
template <int WORDS, typename F, typename B>
__device__ __forceinline__ int32_t cta_hindex(const F& rho, const B& bound, int d, int32_t t, bool direct,
                                              unsigned* bins, int* bounds /* 8 */) {
    if (t <= 0) return 0;
    auto total = [&](int v) {
        const unsigned w = __reduce_add_sync(0xffffffffu, (unsigned)v);
        if ((threadIdx.x & 31) == 0) bounds[threadIdx.x >> 5] = (int)w;
        __syncthreads();
        int tot = 0;
#pragma unroll
        for (int i = 0; i < kThreads / 32; ++i) tot += bounds[i];
        __syncthreads();
        return tot;
    };
    int lo = 0, hi = t, above = 0;
    if (!direct) {
        int cnt = 0, have = 0;
        for (int i = 0; i < d;) {
            const int need = max((min(t - have, 1 << 30) + 4 * kThreads - 1) & ~(4 * kThreads - 1), kCtaSegment);
            const int end = d - i > need ? i + need : d;
            stream_row<kThreads>(rho, i, end, [&](int, int32_t r) { cnt += (r >= t); });
            i = end;
            have = total(cnt);
            if (have >= t) return t;
            if (bound.past(end)) break;
        }
        lo = above = have;
        if (hi - lo <= 1) return lo;
    }
    for (;;) {
        const unsigned span = (unsigned)(hi - lo);
        const int shift = bin_shift(span, WORDS);
        const int nb = (int)((span - 1) >> shift) + 1;
        for (int i = threadIdx.x; i < ((nb + 127) & ~127); i += kThreads) bins[i] = 0;
        __syncthreads();
        int ge = 0, u = hi;  // u: the last bound tested
        for (int i = 0; i < d;) {
            const int end = B::kOn && d - i > kCtaSegment ? i + kCtaSegment : d;
            stream_row<kThreads>(rho, i, end, [&](int, int32_t r) {
                const unsigned x = (unsigned)(r - lo);
                if (x < span) atomicAdd(bins + (x >> shift), 1u);
                else ge += (r >= hi);
            });
            i = end;
            if (!B::kOn || i >= d) continue;
            const int m = max(bound.max_from(i), lo);
            if (m >= u) continue;  // the same for every thread
            u = m;
            __syncthreads();  // the bins so far are complete
            // #{rho >= u} from the bins at or past u
            int c = !F::kCarry || direct ? ge : (threadIdx.x == 0 ? above : 0);
            for (int b = (int)(((unsigned)(u - lo) + (1u << shift) - 1) >> shift) + threadIdx.x; b < nb; b += kThreads)
                c += (int)bins[b];
            if (total(c) >= u) break;
        }
        if (!F::kCarry) {
            above = total(ge);  // with its barriers, the bins are complete too
            if (above >= hi) return hi;
        } else if (direct) {
            above = total(ge);
            if (above >= t) return t;
            direct = false;
        } else {
            __syncthreads();
        }
        if (threadIdx.x < 32) {
            const int b = select_bin<false, WORDS, F::kCarry>(bins, lo, shift, nb, above);
            if (threadIdx.x == 0) {
                bounds[0] = b;
                if (F::kCarry) bounds[1] = above;
            }
        }
        __syncthreads();
        lo += bounds[0] << shift;
        if (F::kCarry) above = bounds[1];
        __syncthreads();
        hi = min(hi, lo + (1 << shift));
        if (hi - lo <= 1) return lo;
    }
}

}  // namespace
